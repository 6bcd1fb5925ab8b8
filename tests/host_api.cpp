// The C ABI's host side without a GPU: the API's sources over a stand-in for
// the CUDA runtime (device memory is host memory, copies are done at once)
// and launches that only note what they were given.  Reads a mesh from the
// file argv[2], runs the check argv[1], prints "ok" and counts.
#include <atomic>
#include <cstdio>
#include <cstdlib>
#include <new>
#include <string>

#include "gks_api.cpp"

// ---- the n-th allocation from here on fails (-1: none)
static std::atomic<long> fail_in{-1};
void* operator new(std::size_t n) {
    if (fail_in.load() >= 0 && fail_in.fetch_sub(1) == 0) throw std::bad_alloc();
    if (void* p = std::malloc(n)) return p;
    throw std::bad_alloc();
}
void operator delete(void* p) noexcept { std::free(p); }
void operator delete(void* p, std::size_t) noexcept { std::free(p); }

// ---- CUDA runtime
static int sm_count = 152;
extern "C" {
cudaError_t cudaMemcpyAsync(void* d, const void* s, size_t n, cudaMemcpyKind, cudaStream_t) {
    std::memmove(d, s, n);
    return cudaSuccess;
}
cudaError_t cudaMemsetAsync(void* d, int v, size_t n, cudaStream_t) {
    std::memset(d, v, n);
    return cudaSuccess;
}
cudaError_t cudaPointerGetAttributes(cudaPointerAttributes* a, const void*) {
    a->type = cudaMemoryTypeDevice;
    return cudaSuccess;
}
cudaError_t cudaStreamCreateWithFlags(cudaStream_t* s, unsigned) { *s = nullptr; return cudaSuccess; }
cudaError_t cudaStreamDestroy(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamBeginCapture(cudaStream_t, cudaStreamCaptureMode) { return cudaSuccess; }
cudaError_t cudaStreamEndCapture(cudaStream_t, cudaGraph_t* g) { *g = nullptr; return cudaSuccess; }
cudaError_t cudaGraphInstantiate(cudaGraphExec_t* e, cudaGraph_t, unsigned long long) { *e = nullptr; return cudaSuccess; }
cudaError_t cudaGraphLaunch(cudaGraphExec_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaGraphDestroy(cudaGraph_t) { return cudaSuccess; }
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t) { return cudaSuccess; }
cudaError_t cudaEventCreate(cudaEvent_t*) { return cudaSuccess; }
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventSynchronize(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float* ms, cudaEvent_t, cudaEvent_t) { *ms = 1.0f; return cudaSuccess; }
cudaError_t cudaGetDevice(int* d) { *d = 3; return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr a, int d) {
    *v = d == 3 && a == cudaDevAttrMultiProcessorCount ? sm_count : -1;
    return cudaSuccess;
}
cudaError_t cudaGetLastError(void) { return cudaSuccess; }
const char* cudaGetErrorString(cudaError_t) { return "error"; }
}

// ---- launches
static int launches = 0;
namespace gks {
static cudaError_t launched() { ++launches; return cudaSuccess; }
template <typename T> cudaError_t Launch<T>::slopes(const DevMesh<T>&, const T*, T*, const Finalize*, cudaStream_t) { return launched(); }
template <typename T> cudaError_t Launch<T>::recon(const DevMesh<T>&, const HostPhys&, const T*, const T*, T*, T*, int32_t*, const Finalize*, int32_t*, cudaStream_t) { return launched(); }
template <typename T> cudaError_t Launch<T>::flux(const DevMesh<T>&, const HostPhys&, const T*, const T*, T*, const double*, double, int, cudaStream_t, int) { return launched(); }
template <typename T> cudaError_t Launch<T>::update1(const DevMesh<T>&, const HostPhys&, const DevState<T>&, cudaStream_t) { return launched(); }
template <typename T> cudaError_t Launch<T>::update2(const DevMesh<T>&, const HostPhys&, const DevState<T>&, cudaStream_t) { return launched(); }
template <typename T> cudaError_t Launch<T>::dt_partials(const DevMesh<T>&, const HostPhys&, const T*, double*, cudaStream_t) { return launched(); }
template <typename T> cudaError_t Launch<T>::pack(const DevMesh<T>&, const HostPhys&, const double*, const double*, T*, double*, unsigned long long*, cudaStream_t, const int32_t*) { return launched(); }
template <typename T> cudaError_t Launch<T>::unpack(const double*, const T*, double*, double*, int64_t, cudaStream_t, const int32_t*) { return launched(); }
template <typename T> cudaError_t Launch<T>::to_double(const T*, double*, int64_t, cudaStream_t) { return launched(); }
template <typename T> cudaError_t Launch<T>::rec_to_double(const DevMesh<T>& m, const T*, const int32_t*, double*, int, const T* X, cudaStream_t) { return m.nf && m.fnw && m.flr && X ? launched() : cudaErrorInvalidValue; }
template <typename T> cudaError_t Launch<T>::poly_to_double(const T*, double*, int64_t, cudaStream_t, const int32_t*) { return launched(); }
template struct Launch<float>;
template struct Launch<double>;
cudaError_t launch_stage(const DevMesh<float>&, const HostPhys&, const DevState<float>&, int, const Launch<float>::Finalize*, unsigned*, cudaStream_t) { return launched(); }
cudaError_t launch_set_control(double*, double*, double*, unsigned long long*, int32_t, double, double, int, int32_t*, cudaStream_t) { return launched(); }
cudaError_t launch_rows_gather(const void*, void*, int64_t, int, const int32_t*, cudaStream_t) { return launched(); }
cudaError_t launch_grid_barrier_probe(unsigned*, int32_t*, int, cudaStream_t) { return launched(); }
cudaError_t launch_wait_probe(int32_t*, int, cudaStream_t) { return launched(); }
cudaError_t adjoint_reverse(const DevMesh<double>&, const HostPhys&, double, const AdjBuffers&, const double*, const double*, const double*, const double*, double*, double*, cudaStream_t) { return launched(); }
int update_blocks(int64_t nc) { return (int)((nc + CELLS_PER_BLOCK - 1) / CELLS_PER_BLOCK); }
}  // namespace gks

#define REQUIRE(x)                                                                                    \
    do {                                                                                              \
        if (!(x)) {                                                                                   \
            std::printf("%s:%d: %s (last error: %s)\n", __FILE__, __LINE__, #x, gks_last_error());    \
            std::exit(1);                                                                             \
        }                                                                                             \
    } while (0)

struct MeshFile {
    std::vector<double> xyz, period;
    std::vector<int64_t> tet;
    std::vector<int8_t> shift, kind;
    int64_t nv = 0, nc = 0;
    explicit MeshFile(const char* path) {
        std::FILE* f = std::fopen(path, "rb");
        REQUIRE(f && std::fread(&nv, 8, 1, f) == 1 && std::fread(&nc, 8, 1, f) == 1);
        xyz.resize(3 * nv);
        period.resize(3);
        tet.resize(4 * nc);
        shift.resize(12 * nc);
        kind.resize(4 * nc);
        REQUIRE(std::fread(xyz.data(), 8, xyz.size(), f) == xyz.size());
        REQUIRE(std::fread(period.data(), 8, 3, f) == 3);
        REQUIRE(std::fread(tet.data(), 8, tet.size(), f) == tet.size());
        REQUIRE(std::fread(shift.data(), 1, shift.size(), f) == shift.size());
        REQUIRE(std::fread(kind.data(), 1, kind.size(), f) == kind.size());
        std::fclose(f);
    }
    gks_mesh* make() const {
        gks_mesh* m = nullptr;
        REQUIRE(gks_mesh_create(xyz.data(), nv, tet.data(), shift.data(), nc, period.data(), &m) == GKS_OK);
        REQUIRE(gks_mesh_set_boundary(m, kind.data()) == GKS_OK);
        REQUIRE(gks_stencil_build(m, nullptr) == GKS_OK);
        return m;
    }
};

static gks_params parameters(int precision, int weno, int constraint = 0) {
    gks_params p;
    gks_params_default(&p);
    p.precision = precision;
    p.weno = weno;
    p.wall_constraint = constraint;
    return p;
}

struct Workspace {
    std::vector<char> raw;
    char* at;
    size_t bytes;
    explicit Workspace(size_t n) : raw(n + 256, 0), bytes(n) {
        at = raw.data() + (256 - (size_t)((uintptr_t)raw.data() & 255)) % 256;
    }
};

// call(): every allocation in turn fails once, until one call has met none;
// check(status) after each.  Returns the number of refused calls.
template <typename Call, typename Check>
static int each_allocation(const Call& call, const Check& check) {
    int refused = 0;
    for (long n = 0;; ++n) {
        gks_status st = GKS_OK;
        bool escaped = false;
        fail_in = n;
        try {
            st = call();
        } catch (...) {
            escaped = true;
        }
        const bool met = fail_in.exchange(-1) < 0;
        REQUIRE(!escaped);
        REQUIRE(st == GKS_OK || st == GKS_E_NOMEM);
        REQUIRE(met || st == GKS_OK);
        check(st);
        refused += st != GKS_OK;
        if (!met) return refused;
    }
}

// what lies outside the staging buffer
static std::string outside_stage(const gks_state* s, const Workspace& w) {
    const size_t a = s->L.stage, b = s->L.cperm ? s->L.cperm : w.bytes;
    return std::string(w.at, w.at + a) + std::string(w.at + b, w.at + w.bytes);
}

static int allocations(const MeshFile& file) {
    int refused = 0;
    gks_mesh* m = nullptr;
    refused += each_allocation(
        [&] { return gks_mesh_create(file.xyz.data(), file.nv, file.tet.data(), file.shift.data(), file.nc, file.period.data(), &m); },
        [&](gks_status st) {
            REQUIRE((m != nullptr) == (st == GKS_OK));
            gks_mesh_destroy(m);
            m = nullptr;
        });
    m = file.make();
    refused += each_allocation([&] { return gks_mesh_set_boundary(m, file.kind.data()); }, [](gks_status) {});
    refused += each_allocation([&] { return gks_stencil_build(m, nullptr); }, [](gks_status) {});
    for (int precision = 0; precision < 3; ++precision) {
        const gks_params p = parameters(precision, 1, precision == 1);
        Workspace w(gks_workspace_bytes(m, &p));
        gks_state* s = nullptr;
        refused += each_allocation([&] { return gks_state_create(m, &p, w.at, w.bytes, nullptr, &s); },
                                   [&](gks_status st) {
                                       REQUIRE((s != nullptr) == (st == GKS_OK));
                                       gks_state_destroy(s);
                                       s = nullptr;
                                   });
        REQUIRE(gks_state_create(m, &p, w.at, w.bytes, nullptr, &s) == GKS_OK);
        s->initialised = true;
        double v[5];
        refused += each_allocation([&] { return gks_timestep(s, v); }, [](gks_status) {});
        refused += each_allocation([&] { return gks_residual(s, v); }, [](gks_status) {});
        // a refused change leaves the device's arrays as they were
        const std::string first = outside_stage(s, w);
        REQUIRE(gks_state_set_variant(s, 1, 2, 0) == GKS_OK);
        const std::string grouped = outside_stage(s, w);
        REQUIRE(gks_state_set_variant(s, 0, 3, 1) == GKS_OK && outside_stage(s, w) == first && grouped != first);
        refused += each_allocation([&] { return gks_state_set_variant(s, 1, 2, 0); }, [&](gks_status st) {
            REQUIRE(outside_stage(s, w) == (st == GKS_OK ? grouped : first));
            REQUIRE(s->flux_variant == (st == GKS_OK ? 0 : 1) && s->slopes_pass == (st == GKS_OK ? 0 : 1));
            REQUIRE(gks_state_set_variant(s, 0, 3, 1) == GKS_OK);
        });
        for (int order = 1; precision > 0 && order < 3; ++order) {
            REQUIRE(gks_state_set_cell_order(s, order) == GKS_OK);
            const std::string there = outside_stage(s, w);
            refused += each_allocation([&] { return gks_state_set_cell_order(s, 0); }, [&](gks_status st) {
                REQUIRE(s->cell_order == (st == GKS_OK ? 0 : order) && s->cperm.empty() == (st == GKS_OK));
                if (st != GKS_OK) REQUIRE(outside_stage(s, w) == there);
                REQUIRE(gks_state_set_cell_order(s, order) == GKS_OK && outside_stage(s, w) == there);
            });
            REQUIRE(gks_state_set_cell_order(s, 0) == GKS_OK);
            refused += each_allocation([&] { return gks_state_set_cell_order(s, order); }, [&](gks_status st) {
                REQUIRE(s->cell_order == (st == GKS_OK ? order : 0) && s->cinv.empty() == (st != GKS_OK));
                REQUIRE(gks_state_set_cell_order(s, 0) == GKS_OK);
            });
        }
        gks_state_destroy(s);
    }
    gks_mesh_destroy(m);
    return refused;
}

// the arrays of one state against the mesh, element by element
template <typename T, typename TO>
static void compare_arrays(const gks_state* s, const gks_mesh& g) {
    const Layout& L = s->L;
    const int64_t nc = g.nc, nf = g.nf, nblk = update_blocks(nc);
    auto i32 = [&](size_t off) { return reinterpret_cast<const int32_t*>(s->ws + off); };
    const TO* tile = reinterpret_cast<const TO*>(s->ws + L.tile);
    const T* fgeo = reinterpret_cast<const T*>(s->ws + L.fgeo);
    const T* fnw = reinterpret_cast<const T*>(s->ws + L.fnw);
    const int32_t *perm = i32(L.perm), *flr = i32(L.flr), *cface = i32(L.cface);
    auto pub = [&](int64_t d) { return s->cperm.empty() ? d : (int64_t)s->cperm[d]; };
    for (int64_t d = 0; d < nblk * CELLS_PER_BLOCK; ++d) {
        const TO* blk = tile + d / CELLS_PER_BLOCK * TILE_ROWS * CELLS_PER_BLOCK;
        auto row = [&](int r) { return blk[tile_at<TO>(r, (int)(d % CELLS_PER_BLOCK))]; };
        if (d >= nc) {
            for (int r = 0; r < TILE_ROWS; ++r) REQUIRE(row(r) == TO(0));
            continue;
        }
        const int64_t c = pub(d);
        double far[3] = {0.0, 0.0, 0.0};
        for (int k = 0; k < 144; ++k) REQUIRE(row(TILE_M2 + k) == (TO)g.M2[c * 144 + k]);
        for (int k = 0; k < 12; ++k) REQUIRE(row(TILE_M1 + k) == (TO)g.M1[c * 12 + k]);
        for (int k = 0; k < 6; ++k) REQUIRE(row(TILE_MOM + k) == (TO)g.mom2[c * 6 + k]);
        REQUIRE(row(TILE_V23) == (TO)std::pow(g.vol[c], 2.0 / 3.0) && row(TILE_V43) == (TO)std::pow(g.vol[c], 4.0 / 3.0));
        for (int f = 0; f < 4; ++f) {
            const int64_t face = g.csr_face[c * 4 + f];
            const bool left = g.csr_sign[c * 4 + f] > 0;
            const int32_t e = cface[f * nc + d];
            REQUIRE(perm[e >> 1] == face && (e & 1) == (left ? 0 : 1));
            REQUIRE(flr[(left ? 0 : nf) + (e >> 1)] == (int32_t)d);
            for (int k = 0; k < 9; ++k) {
                const double x = (left ? g.gp_l : g.gp_r)[face * 9 + k];
                REQUIRE(row(TILE_G + f * 9 + k) == (TO)x);
                REQUIRE(fgeo[(e >> 1) * FGEO + (left ? 4 : 13) + k] == (T)x);
                if (std::abs(x) > far[k % 3]) far[k % 3] = std::abs(x);
            }
            if (g.nbr[c * 4 + f] < 0) REQUIRE(flr[(left ? nf : 0) + (e >> 1)] == -1 - (int32_t)s->bkind[face]);
        }
        for (int k = 0; k < 3; ++k) REQUIRE(row(TILE_BND + k) == (TO)far[k]);
    }
    for (int64_t d = 0; d < nf; ++d) {
        const int64_t f = perm[d];
        for (int k = 0; k < 4; ++k) {
            const T v = k < 3 ? (T)g.fnorm[f * 3 + k] : (T)(g.farea[f] / 3.0);
            REQUIRE(fgeo[d * FGEO + k] == v && fnw[d * 4 + k] == v);
        }
        for (int k = 0; L.fan && k < 3; ++k) {
            const float* a = reinterpret_cast<const float*>(s->ws + L.fan) + 6 * d + 2 * k;
            const double v = g.farea[f] * g.fnorm[f * 3 + k];
            REQUIRE(a[0] == (float)v && a[1] == (float)(v - (double)(float)v));
        }
    }
}

static int arrays(const MeshFile& file) {
    int states = 0;
    gks_mesh* m = file.make();
    for (int precision = 0; precision < 3; ++precision)
        for (int cells = 0; cells < (precision ? 3 : 1); ++cells)
            for (int faces = 0; faces < 2; ++faces, ++states) {
                const gks_params p = parameters(precision, 1);
                Workspace w(gks_workspace_bytes(m, &p));
                std::memset(w.at, 0x55, w.bytes);
                gks_state* s = nullptr;
                REQUIRE(gks_state_create(m, &p, w.at, w.bytes, nullptr, &s) == GKS_OK);
                if (cells) REQUIRE(gks_state_set_cell_order(s, cells) == GKS_OK);
                REQUIRE(gks_state_set_variant(s, faces, 3, 1) == GKS_OK);
                // the records' conversion has the mesh and the state it reads
                s->initialised = true;
                for (int stage = 1; stage < 3; ++stage)
                    REQUIRE(gks_debug_face_records(s, 0.1, stage, reinterpret_cast<double*>(w.at)) == GKS_OK);
                if (precision == 0) compare_arrays<double, double>(s, *m);
                if (precision == 1) compare_arrays<float, float>(s, *m);
                if (precision == 2) compare_arrays<float, double>(s, *m);
                gks_state_destroy(s);
            }
    gks_mesh_destroy(m);
    return states;
}

// the mesh's boundary kinds change after a state's creation: the state keeps
// its own through every re-upload, and takes no fixed state it has no room for
static int kinds(const MeshFile& file) {
    int states = 0;
    for (int precision = 0; precision < 3; ++precision)
        for (int constraint = 0; constraint < 2; ++constraint)
            for (int kind = GKS_BC_OPEN; kind <= GKS_BC_MOVING_WALL; ++kind, ++states) {
                gks_mesh* m = file.make();
                const gks_params p = parameters(precision, 1, constraint);
                Workspace w(gks_workspace_bytes(m, &p));
                gks_state* s = nullptr;
                REQUIRE(gks_state_create(m, &p, w.at, w.bytes, nullptr, &s) == GKS_OK);
                const std::string first = outside_stage(s, w);
                const std::vector<int8_t> later(file.kind.size(), (int8_t)kind);
                REQUIRE(gks_mesh_set_boundary(m, later.data()) == GKS_OK);
                REQUIRE(gks_state_set_variant(s, 1, 3, 1) == GKS_OK && gks_state_set_variant(s, 0, 3, 1) == GKS_OK);
                REQUIRE(outside_stage(s, w) == first);
                if (precision) {
                    REQUIRE(gks_state_set_cell_order(s, 2) == GKS_OK && gks_state_set_cell_order(s, 0) == GKS_OK);
                    // (the order's own two arrays, right after the staging buffer, keep what they held)
                    const size_t orders = 2 * ((4 * (size_t)m->nc + 255) & ~(size_t)255), at = first.size();
                    const std::string now = outside_stage(s, w);
                    const size_t a = s->L.stage, b = a + orders;
                    REQUIRE(now.substr(0, a) == first.substr(0, a) && now.substr(b, at) == first.substr(b, at));
                }
                const int before = launches;
                std::vector<double> W(20 * (size_t)m->nc, 1.0);
                REQUIRE(gks_set_fixed_state(s, W.data(), W.data()) == GKS_E_ARG && launches == before);
                gks_state_destroy(s);
                gks_mesh_destroy(m);
            }
    return states;
}

// the adjoint's scratch is read and written in 16-byte vectors
static int scratch(const MeshFile& file) {
    gks_mesh* m = file.make();
    const gks_params p = parameters(0, 1);
    Workspace w(gks_workspace_bytes(m, &p));
    gks_state* s = nullptr;
    REQUIRE(gks_state_create(m, &p, w.at, w.bytes, nullptr, &s) == GKS_OK);
    const size_t bytes = gks_adjoint_workspace_bytes(s);
    Workspace room(bytes + 256);
    std::vector<double> v(20 * (size_t)m->nc, 1.0);
    double* d = v.data();
    int refused = 0;
    for (size_t off = 0; off < 32; off += 8) {
        const int before = launches;
        const gks_status a = gks_adjoint_step(s, 0.1, d, d, d, d, d, d, room.at + off, bytes);
        const gks_status b = gks_adjoint_step_staged(s, 0.1, d, d, d, d, d, d, d, d, room.at + off, bytes);
        REQUIRE(a == (off % 16 ? GKS_E_ARG : GKS_OK) && b == a);
        REQUIRE((launches == before) == (off % 16 != 0));
        refused += a != GKS_OK;
    }
    gks_state_destroy(s);
    gks_mesh_destroy(m);
    return refused;
}

// a state that made no step has no residual, whatever its workspace held
static int residual(const MeshFile& file) {
    gks_mesh* m = file.make();
    int zeros = 0;
    for (int precision = 0; precision < 3; ++precision) {
        const gks_params p = parameters(precision, 1);
        Workspace w(gks_workspace_bytes(m, &p));
        std::memset(w.at, 0xff, w.bytes);  // every double a NaN
        gks_state* s = nullptr;
        REQUIRE(gks_state_create(m, &p, w.at, w.bytes, nullptr, &s) == GKS_OK);
        s->initialised = true;
        double dt, r[5];
        REQUIRE(gks_timestep(s, &dt) == GKS_OK && gks_residual(s, r) == GKS_OK);
        for (double v : r) zeros += v == 0.0;
        gks_state_destroy(s);
    }
    gks_mesh_destroy(m);
    return zeros;
}

// the FP64 flux's blocks follow the device's own number of SMs
static int flux_blocks(const MeshFile& file) {
    gks_mesh* m = file.make();
    int small = 0;
    for (int sms : {1, 2, 76, 132, 148, 152, 160}) {
        sm_count = sms;
        for (int precision = 0; precision < 2; ++precision) {
            const gks_params p = parameters(precision, 1);
            Workspace w(gks_workspace_bytes(m, &p));
            gks_state* s = nullptr;
            REQUIRE(gks_state_create(m, &p, w.at, w.bytes, nullptr, &s) == GKS_OK);
            REQUIRE((precision ? s->m32.sms : s->m64.sms) == sms);
            gks_state_destroy(s);
        }
        // the blocks of a launch dealt to the SMs in turn
        for (int64_t nf = 1; nf < 60000; nf = nf * 5 / 4 + 1) {
            int64_t most[2] = {0, 0};
            for (int small_blocks = 0; small_blocks < 2; ++small_blocks) {
                const int faces = small_blocks ? 21 : 32, warps = small_blocks ? 2 : 3;
                std::vector<int64_t> load((size_t)sms, 0);
                for (int64_t f = 0, b = 0; f < nf; f += faces, ++b) load[(size_t)(b % sms)] += warps;
                for (int64_t v : load) most[small_blocks] = std::max(most[small_blocks], v);
            }
            REQUIRE(flux_small_blocks(nf, sms) == (most[1] < most[0]));
            small += most[1] < most[0];
        }
    }
    sm_count = 152;
    gks_mesh_destroy(m);
    return small;
}

int main(int argc, char** argv) {
    REQUIRE(argc == 3);
    const std::string check = argv[1];
    const MeshFile file(argv[2]);
    if (check == "allocations") {
        std::printf("ok %d\n", allocations(file));
        return 0;
    }
    if (check == "kinds") {
        std::printf("ok %d\n", kinds(file));
        return 0;
    }
    if (check == "scratch") {
        std::printf("ok %d\n", scratch(file));
        return 0;
    }
    if (check == "residual") {
        std::printf("ok %d\n", residual(file));
        return 0;
    }
    if (check == "flux_blocks") {
        std::printf("ok %d\n", flux_blocks(file));
        return 0;
    }
    if (check == "arrays") {
        std::printf("ok %d\n", arrays(file));
        return 0;
    }
    std::printf("unknown check %s\n", argv[1]);
    return 1;
}

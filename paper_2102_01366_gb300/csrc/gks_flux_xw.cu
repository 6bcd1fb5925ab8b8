// gks_flux_xw.cu -- the face-flux instances for meshes with isothermal or
// moving wall faces (Sec. 4.4 ghosts of those walls compiled in), kept apart
// so that the common instances carry no code for them and the two sets
// compile in parallel.
#include <cuda_runtime.h>

#include "gks_flux.cuh"

namespace gks {

template <typename T>
cudaError_t launch_flux_xw(const DevMesh<T>& m, const HostPhys& p, const T* W, const T* poly, T* rec,
                           const double* ctrl, double dt_override, int stage, cudaStream_t s, int variant) {
    return launch_flux<T, true>(m, p, W, poly, rec, ctrl, dt_override, stage, s, variant);
}

template cudaError_t launch_flux_xw(const DevMesh<double>&, const HostPhys&, const double*, const double*, double*,
                                    const double*, double, int, cudaStream_t, int);
template cudaError_t launch_flux_xw(const DevMesh<float>&, const HostPhys&, const float*, const float*, float*,
                                    const double*, double, int, cudaStream_t, int);

}  // namespace gks

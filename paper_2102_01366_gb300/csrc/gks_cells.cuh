// gks_cells.cuh -- lane layout of the cell kernels, shared by the
// translation units that hold them.
#pragma once

#include <cstdint>

#include "gks_kernels.h"

namespace gks {

// a barrier of `count` threads on named barrier `id` (0: the whole block)
__device__ __forceinline__ void group_barrier(int id, int count) {
    if (id == 0)
        __syncthreads();
    else
        asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(count) : "memory");
}

// N values (N a multiple of the vector's length) from 16-byte aligned memory
template <int N, typename T>
__device__ __forceinline__ void load_vec(const T* __restrict__ p, T* v) {
    if constexpr (sizeof(T) == 4) {
        static_assert(N % 4 == 0, "whole vectors");
#pragma unroll
        for (int i = 0; i < N / 4; ++i) {
            const float4 x = reinterpret_cast<const float4*>(p)[i];
            v[4 * i] = x.x;
            v[4 * i + 1] = x.y;
            v[4 * i + 2] = x.z;
            v[4 * i + 3] = x.w;
        }
    } else {
        static_assert(N % 2 == 0, "whole vectors");
#pragma unroll
        for (int i = 0; i < N / 2; ++i) {
            const double2 x = reinterpret_cast<const double2*>(p)[i];
            v[2 * i] = x.x;
            v[2 * i + 1] = x.y;
        }
    }
}

template <int N, typename T>
__device__ __forceinline__ void store_vec(T* __restrict__ p, const T* v) {
    if constexpr (sizeof(T) == 4) {
#pragma unroll
        for (int i = 0; i < N / 4; ++i)
            reinterpret_cast<float4*>(p)[i] = make_float4(v[4 * i], v[4 * i + 1], v[4 * i + 2], v[4 * i + 3]);
    } else {
#pragma unroll
        for (int i = 0; i < N / 2; ++i) reinterpret_cast<double2*>(p)[i] = make_double2(v[2 * i], v[2 * i + 1]);
    }
}

// 5 lanes per cell (one per conservative component), 6 cells per warp (lanes
// 30, 31 idle), CELLS_PER_BLOCK cells per 128-thread block
struct CellLane {
    int64_t c;    // cell (clamped to a valid cell on idle lanes)
    int q;        // component
    int base;     // lane of component 0 of this cell
    bool active;  // lane carries a real (cell, component)
};

// vb: the block of CELLS_PER_BLOCK cells, tid: the thread within its
// CELL_THREADS
__device__ __forceinline__ CellLane cell_lane(int64_t nc, int64_t vb, int tid) {
    CellLane L;
    const int lane = tid & 31;
    const int warp = tid >> 5;
    const int cl = lane / 5;
    L.q = lane - 5 * cl;
    L.base = lane - L.q;
    const int64_t c = vb * CELLS_PER_BLOCK + warp * 6 + cl;
    L.active = lane < 30 && c < nc;
    L.c = c < nc ? c : nc - 1;
    return L;
}

static inline unsigned cell_grid(int64_t nc) { return (unsigned)((nc + CELLS_PER_BLOCK - 1) / CELLS_PER_BLOCK); }

}  // namespace gks

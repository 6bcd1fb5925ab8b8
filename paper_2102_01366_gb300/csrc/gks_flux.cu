// gks_flux.cu -- face flux kernels (Sec. 2.2, 3, 4.4, 4.5), sm_103a, FP64 and
// FP32-bulk instantiations.
//
//   k_flux  face-ordered, one thread per Gauss point: R of both cells at the
//           point, face frame, kinetic solution (Eq. 2nd-flux with the
//           equilibrium state of Eq. new-equ-part), weighted face record of
//           the stage (Sec. 3 Eqs. linear-system, s2o4, step-du)
//
// Boundary faces take their ghost side from the face's kind (Sec. 4.4 slip
// wall, a fixed state, or zeroth-order extrapolation).
#include <cuda_runtime.h>

#include "gks_flux.cuh"

namespace gks {

template <typename T>
cudaError_t Launch<T>::flux(const DevMesh<T>& m, const HostPhys& p, const T* W, const T* poly, T* rec,
                            const double* ctrl, double dt_override, int stage, cudaStream_t s, int variant) {
    // ctrl is the per-case step array (NULL: dt_override everywhere)
    if (m.nf == 0) return cudaSuccess;
    if (m.xwalls) return launch_flux_xw(m, p, W, poly, rec, ctrl, dt_override, stage, s, variant);
    return launch_flux<T, false>(m, p, W, poly, rec, ctrl, dt_override, stage, s, variant);
}

template cudaError_t Launch<double>::flux(const DevMesh<double>&, const HostPhys&, const double*, const double*,
                                          double*, const double*, double, int, cudaStream_t, int);
template cudaError_t Launch<float>::flux(const DevMesh<float>&, const HostPhys&, const float*, const float*,
                                         float*, const double*, double, int, cudaStream_t, int);

}  // namespace gks

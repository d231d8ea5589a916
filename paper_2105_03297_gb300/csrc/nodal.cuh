// Nodal-state form of the projected CG.  Every CG vector of the strain form
// is compatible (it lies in the range of G = B K^-1 B^T, K = B^T B), so it is B
// applied to a nodal field: x = B xi, r = B rho, p = B pi, and q = G C p = B w
// with w = K^-1 B^T C B pi.  Running the same CG on the nodal fields (D
// components per node instead of m per voxel) gives the same iterates; the
// inner products stay those of the strain space:
//   <p, C p> = sum over elements of (B pi) : C (B pi)
//   <r, r>   = |B rho|^2 = <rho, K rho> = <rho, R>
// This is the preconditioned-FE reading of the projection (Sec. 4: the
// operator acts as a preconditioner of the FE stiffness with B^T B in the
// role of the reference stiffness).  The residual kept from iteration to
// iteration is the force R = K rho, as x-transformed spectra: it is updated
// where the force spectra are loaded, and rho = K^-1 R and <rho, R> come out of
// the solve per wavevector, so that no pass over real space is needed between
// the last pass of one iteration and the first of the next.
//
//   first pass (pass_force.cuh)  pi = rho + beta pi_old, xi += alpha_prev
//                                pi_old, f = B^T C B pi, <B pi, C B pi> -> alpha
//   pass B (2D: C)               R -= alpha f
//   pass C                       rho^ = (B^H B)^-1 R^, <rho, R> -> beta
//   passes D, E                  rho
// Measured at 256^3 in FP32: the separate update kernel (rho -= alpha w and
// |B rho|^2 by the element stencils) took 0.24 of 1.9 ms per iteration.
//
// pi alternates between two buffers (the first pass reads its neighbours' old
// values while owners write new ones).
#pragma once
#include "pass3d.cuh"

namespace rve {

// After the CG: xi += alpha pi_last (the deferred update, for load cases that
// ran an iteration and did not break down), then u += xi in FP64.
// grid (ceil(N / NT), L).  pi_even / pi_odd: direction buffers of even / odd
// iterations.
template <typename T, int NT>
__global__ void __launch_bounds__(NT) nodal_finish(PassArgs<T> a, const T* __restrict__ pi_even,
                                                   const T* __restrict__ pi_odd, const T* __restrict__ xi) {
  const int l = blockIdx.y;
  const CgState* cg = a.cg + l;
  if (!cg->active) return;
  const int64_t N = a.N;
  const int64_t v = (int64_t)blockIdx.x * NT + threadIdx.x;
  if (v >= N) return;
  const bool last = cg->it > 0 && cg->status != ST_BAD;
  const T alpha = last ? cg_alpha<T>(cg) : (T)0;
  const T* pl = ((cg->it - 1) & 1) ? pi_odd : pi_even;
  const int64_t lbase = (int64_t)l * a.dim * N;
  for (int j = 0; j < a.dim; ++j) {
    T x = xi[lbase + j * N + v];
    if (last) x += alpha * pl[lbase + j * N + v];
    a.u64[lbase + j * N + v] += (double)x;
  }
}

// ------------------------------------------------------------ launchers
template <typename T>
cudaError_t launch_nodal_finish(const PassArgs<T>& a, const T* pi_even, const T* pi_odd, const T* xi,
                                cudaStream_t s) {
  constexpr int NT = 256;
  dim3 grid((unsigned)((a.N + NT - 1) / NT), a.L);
  nodal_finish<T, NT><<<grid, NT, 0, s>>>(a, pi_even, pi_odd, xi);
  return cudaGetLastError();
}

}  // namespace rve

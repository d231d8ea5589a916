// Nodal-state form of the projected CG.  Every CG vector of the strain form
// is compatible (it lies in the range of G = B K^-1 B^T), so it is B applied
// to a nodal field: x = B xi, r = B rho, p = B pi, and q = G C p = B w with
// w = K^-1 B^T C B pi.  Running the same CG on the nodal fields (D
// components per node instead of m per voxel) gives the same iterates; the
// inner products stay those of the strain space:
//   <p, C p> = sum over elements of (B pi) : C (B pi)     (force kernel)
//   <r, r>   = sum over elements of |B rho|^2              (update kernel)
// This is the preconditioned-FE reading of the projection (Sec. 4: the
// operator acts as a preconditioner of the FE stiffness with B^T B in the
// role of the reference stiffness).
//
//   first pass     pi = rho + beta pi_old, xi += alpha_prev pi_old,
//                  f = B^T C B pi, <B pi, C B pi> -> alpha (pass_force.cuh)
//   FFT passes     w = F^-1 (B^H B)^-1 F f    (D components)
//   update kernel  rho_new = rho - alpha w, <B rho_new, B rho_new> -> beta
//
// pi and rho each alternate between two buffers (the kernels read their
// neighbours' old values while owners write new ones).
#pragma once
#include "pass3d.cuh"

namespace rve {

// ----------------------------------------------------------------- 3D
// Mandel strains of the six tetrahedra of a voxel from its corner
// displacements uc[c][j], corner c = dx + 2 dy + 4 dz.
template <typename T>
__device__ __forceinline__ void tet_strains_3d(const T uc[8][3], const T* ih, T* pv /*[36]*/) {
  const T r2 = (T)kInvSqrt2;
#pragma unroll
  for (int t = 0; t < 6; ++t) {
    const int pa = kuhn_perm(t, 0), pb = kuhn_perm(t, 1), pc = kuhn_perm(t, 2);
    const int v1 = 1 << pa, v2 = v1 | (1 << pb);
    T H[3][3];
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      H[pa][j] = (uc[v1][j] - uc[0][j]) * ih[pa];
      H[pb][j] = (uc[v2][j] - uc[v1][j]) * ih[pb];
      H[pc][j] = (uc[7][j] - uc[v2][j]) * ih[pc];
    }
    T* q = pv + 6 * t;
    q[0] = H[0][0]; q[1] = H[1][1]; q[2] = H[2][2];
    q[3] = r2 * (H[1][2] + H[2][1]);
    q[4] = r2 * (H[0][2] + H[2][0]);
    q[5] = r2 * (H[0][1] + H[1][0]);
  }
}

// rho_new = rho_old - alpha w (init: rho = -w, xi = 0) at every node and
// <B rho_new, B rho_new> over the six tetrahedra of every voxel.  Thread
// (x, y) sweeps z over a chunk of kUZ planes, keeping the updated corner
// values of plane z + 1 for the next step; the node (x, y, z) is written
// once.  NT threads cover bx x by columns, bx = min(n_x, 32), by = NT / bx;
// grid (n_x/bx, n_y/by, (n_z/kUZ) L).
constexpr int kUZ = 16;
template <typename T, int NT>
__global__ void __launch_bounds__(NT) nodal_update_3d(PassArgs<T> a, const T* __restrict__ rho_old,
                                                      const T* __restrict__ w, T* __restrict__ rho_new,
                                                      T* __restrict__ xi, int init) {
  __shared__ double red[NT / 32];
  __shared__ int flag;
  const int nx = a.n[0], ny = a.n[1], nz = a.n[2];
  const int tz = nz < kUZ ? nz : kUZ;
  const int nzc = nz / tz;
  const int l = blockIdx.z / nzc, zc = blockIdx.z % nzc;
  CgState* cg = a.cg + l;
  if (!cg->active) return;
  if (a.cgphase && cg->status != ST_RUN) return;
  const int64_t N = a.N;
  const int bx = nx < 32 ? nx : 32, by = NT / bx;
  const int x = blockIdx.x * bx + (threadIdx.x & (bx - 1)), y = blockIdx.y * by + threadIdx.x / bx;
  const int x1 = (x + 1) & (nx - 1), y1 = (y + 1) & (ny - 1);
  const T alpha = init ? (T)0 : cg_alpha<T>(cg);
  const int64_t lbase = (int64_t)l * 3 * N;
  const int64_t plane = (int64_t)nx * ny;
  const int64_t o00 = (int64_t)y * nx + x, o10 = (int64_t)y * nx + x1;
  const int64_t o01 = (int64_t)y1 * nx + x, o11 = (int64_t)y1 * nx + x1;
  const int z0 = zc * tz;
  // updated values of the 4 corners (dx, dy) of one node plane
  auto corners = [&](int z, T c[4][3]) {
    const int64_t pb = lbase + (int64_t)(z & (nz - 1)) * plane;
    const int64_t off[4] = {o00, o10, o01, o11};
#pragma unroll
    for (int k = 0; k < 4; ++k)
#pragma unroll
      for (int j = 0; j < 3; ++j) {
        const int64_t i = pb + (int64_t)j * N + off[k];
        c[k][j] = init ? -__ldg(w + i) : __ldg(rho_old + i) - alpha * __ldg(w + i);
      }
  };
  T lo[4][3], hi[4][3];
  corners(z0, lo);
  T acc = 0;
  for (int z = z0; z < z0 + tz; ++z) {
    corners(z + 1, hi);
    const int64_t v = lbase + (int64_t)z * plane + o00;
#pragma unroll
    for (int j = 0; j < 3; ++j) rho_new[v + (int64_t)j * N] = lo[0][j];
    if (init) {
#pragma unroll
      for (int j = 0; j < 3; ++j) xi[v + (int64_t)j * N] = 0;
    }
    T uc[8][3];
#pragma unroll
    for (int k = 0; k < 4; ++k)
#pragma unroll
      for (int j = 0; j < 3; ++j) { uc[k][j] = lo[k][j]; uc[k + 4][j] = hi[k][j]; }
    T pv[36];
    tet_strains_3d<T>(uc, a.ih, pv);
#pragma unroll
    for (int c = 0; c < 36; ++c) acc += pv[c] * pv[c];
#pragma unroll
    for (int k = 0; k < 4; ++k)
#pragma unroll
      for (int j = 0; j < 3; ++j) lo[k][j] = hi[k][j];
  }
  const double s = block_sum<NT>((double)acc, red);
  const int nblk = gridDim.x * gridDim.y * nzc;
  const int blk = blockIdx.x + gridDim.x * (blockIdx.y + gridDim.y * zc);
  double* part = a.part + (int64_t)l * a.part_stride;
  if (publish_partial(s, part, &cg->cnt_e, blk, nblk, &flag)) {
    const double rr = sum_partials<NT>(part, nblk, red);
    if (threadIdx.x == 0) finish_rr(cg, rr, init != 0);
  }
}

// ----------------------------------------------------------------- 2D
// Mandel strains of the two triangles of a pixel from its corner
// displacements uc[c][j], corner c = dx + 2 dy.
template <typename T>
__device__ __forceinline__ void tri_strains_2d(const T uc[4][2], T ihx, T ihy, T* q /*[6]*/) {
  const T r2 = (T)kInvSqrt2;
  // element 0 = nodes {00, 10, 01}; element 1 = nodes {11, 01, 10}
  q[0] = (uc[1][0] - uc[0][0]) * ihx;
  q[1] = (uc[2][1] - uc[0][1]) * ihy;
  q[2] = r2 * ((uc[2][0] - uc[0][0]) * ihy + (uc[1][1] - uc[0][1]) * ihx);
  q[3] = (uc[3][0] - uc[2][0]) * ihx;
  q[4] = (uc[3][1] - uc[1][1]) * ihy;
  q[5] = r2 * ((uc[3][0] - uc[1][0]) * ihy + (uc[3][1] - uc[2][1]) * ihx);
}

// 2D counterpart of nodal_update_3d: NT threads cover bx columns (bx =
// min(n_x, NT)) x NT/bx row groups of kUY rows; each thread sweeps its rows
// keeping the updated corner values of row y + 1.  grid (n_x/bx,
// max(1, n_y/(kUY NT/bx)) L); row groups past n_y are idle.
constexpr int kUY = 16;
template <typename T, int NT>
__global__ void __launch_bounds__(NT) nodal_update_2d(PassArgs<T> a, const T* __restrict__ rho_old,
                                                      const T* __restrict__ w, T* __restrict__ rho_new,
                                                      T* __restrict__ xi, int init) {
  __shared__ double red[NT / 32];
  __shared__ int flag;
  const int nx = a.n[0], ny = a.n[1];
  const int bx = nx < NT ? nx : NT, by = NT / bx;
  const int rows_blk = by * kUY;
  const int nyb = ny > rows_blk ? ny / rows_blk : 1;
  const int l = blockIdx.y / nyb, yb = blockIdx.y % nyb;
  CgState* cg = a.cg + l;
  if (!cg->active) return;
  if (a.cgphase && cg->status != ST_RUN) return;
  const int64_t N = a.N;
  const int x = blockIdx.x * bx + (threadIdx.x % bx);
  const int ys = yb * rows_blk + (threadIdx.x / bx) * kUY;
  const int x1 = (x + 1) & (nx - 1);
  const T alpha = init ? (T)0 : cg_alpha<T>(cg);
  const int64_t lbase = (int64_t)l * 2 * N;
  T acc = 0;
  if (ys < ny) {
    auto corners = [&](int y, T c[2][2]) {
      const int64_t rb = lbase + (int64_t)(y & (ny - 1)) * nx;
#pragma unroll
      for (int j = 0; j < 2; ++j) {
        const int64_t i0 = rb + (int64_t)j * N + x, i1 = rb + (int64_t)j * N + x1;
        c[0][j] = init ? -__ldg(w + i0) : __ldg(rho_old + i0) - alpha * __ldg(w + i0);
        c[1][j] = init ? -__ldg(w + i1) : __ldg(rho_old + i1) - alpha * __ldg(w + i1);
      }
    };
    T lo[2][2], hi[2][2];
    corners(ys, lo);
    for (int y = ys; y < ys + kUY; ++y) {
      corners(y + 1, hi);
      const int64_t v = lbase + (int64_t)y * nx + x;
      rho_new[v] = lo[0][0];
      rho_new[v + N] = lo[0][1];
      if (init) { xi[v] = 0; xi[v + N] = 0; }
      const T uc[4][2] = {{lo[0][0], lo[0][1]}, {lo[1][0], lo[1][1]}, {hi[0][0], hi[0][1]}, {hi[1][0], hi[1][1]}};
      T q[6];
      tri_strains_2d<T>(uc, a.ih[0], a.ih[1], q);
#pragma unroll
      for (int c = 0; c < 6; ++c) acc += q[c] * q[c];
#pragma unroll
      for (int k = 0; k < 2; ++k) { lo[k][0] = hi[k][0]; lo[k][1] = hi[k][1]; }
    }
  }
  const double s = block_sum<NT>((double)acc, red);
  const int nblk = gridDim.x * nyb;
  const int blk = blockIdx.x + gridDim.x * yb;
  double* part = a.part + (int64_t)l * a.part_stride;
  if (publish_partial(s, part, &cg->cnt_e, blk, nblk, &flag)) {
    const double rr = sum_partials<NT>(part, nblk, red);
    if (threadIdx.x == 0) finish_rr(cg, rr, init != 0);
  }
}

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
cudaError_t launch_nodal_update(const PassArgs<T>& a, const T* rho_old, const T* w, T* rho_new, T* xi, int init,
                                cudaStream_t s) {
  constexpr int NT = 256;
  if (a.dim == 3) {
    const int bx = a.n[0] < 32 ? a.n[0] : 32, by = NT / bx;   // n_y >= 16 >= by
    const int tz = a.n[2] < kUZ ? a.n[2] : kUZ;
    dim3 grid(a.n[0] / bx, a.n[1] / by, (a.n[2] / tz) * a.L);
    nodal_update_3d<T, NT><<<grid, NT, 0, s>>>(a, rho_old, w, rho_new, xi, init);
  } else {
    const int bx = a.n[0] < NT ? a.n[0] : NT, rows_blk = (NT / bx) * kUY;
    const int nyb = a.n[1] > rows_blk ? a.n[1] / rows_blk : 1;
    dim3 grid(a.n[0] / bx, nyb * a.L);
    nodal_update_2d<T, NT><<<grid, NT, 0, s>>>(a, rho_old, w, rho_new, xi, init);
  }
  return cudaGetLastError();
}

template <typename T>
cudaError_t launch_nodal_finish(const PassArgs<T>& a, const T* pi_even, const T* pi_odd, const T* xi,
                                cudaStream_t s) {
  constexpr int NT = 256;
  dim3 grid((unsigned)((a.N + NT - 1) / NT), a.L);
  nodal_finish<T, NT><<<grid, NT, 0, s>>>(a, pi_even, pi_odd, xi);
  return cudaGetLastError();
}

}  // namespace rve

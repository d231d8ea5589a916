// 3D projected-operator passes (six Kuhn tetrahedra per voxel).
//
// Real fields are [l][c][z][y][x].  One application of q = G * (C : p):
//   A  force pass (pass_force.cuh): material, CG direction update, <p, C p>,
//      nodal forces t = B^H sigma in real space, forward real FFT along x;
//      writes spec1 as [l][j][k_x][z][y] (y contiguous), two partial sums of
//      t (planes z and z + 1) for each of the D = 3 nodal components j;
//   B  their sum and its forward FFT along y; writes spec2 as [l][j][k_x][k_y][z]
//      (z contiguous, chunks of TZB z per k_y);
//   C  forward FFT along z, w^ = (B^H B)^-1 t^ per wavevector, inverse FFT
//      along z, in place on spec2;
//   D  inverse FFT along y, spec2 -> spec1;
//   E  inverse real FFT along x of w, q = B w in real space, r -= alpha q,
//      <r, r> (x += alpha p is deferred to the next pass A, as in 2D).
// Tile variant 5 (pass3d_pipe.cuh) transforms all 36 stress components along x
// instead, and B forms t from them (differences along y and z).
// The other derivatives (one evaluation point) and finite strain carry all
// their components through B, C (with the projection), D and E.
// Measured at 256 x 256 x 64, one load case, FP32, us per iteration: all 36
// components through every pass A 656, B 168, C 371, D 184, E 388; the nodal
// ones A 622, B 38, C 50, D 28, E 297.
#pragma once
#include "pass2d.cuh"
#include "pass3d_pipe.cuh"

namespace rve {

// Kuhn tetrahedron Theta = permutation (a, b, c) of (x, y, z), lexicographic.
__host__ __device__ constexpr int kuhn_perm(int t, int i) {
  // rows: (0,1,2) (0,2,1) (1,0,2) (1,2,0) (2,0,1) (2,1,0)
  return (t == 0) ? (i == 0 ? 0 : i == 1 ? 1 : 2)
       : (t == 1) ? (i == 0 ? 0 : i == 1 ? 2 : 1)
       : (t == 2) ? (i == 0 ? 1 : i == 1 ? 0 : 2)
       : (t == 3) ? (i == 0 ? 1 : i == 1 ? 2 : 0)
       : (t == 4) ? (i == 0 ? 2 : i == 1 ? 0 : 1)
                  : (i == 0 ? 2 : i == 1 ? 1 : 0);
}

// --------------------------------------------- L2 prefetch of a later tile
// The transform passes run grids of far more blocks than are resident, and
// the blocks start in about linear launch order as earlier ones retire.  With
// a.pf_ahead = D > 0 every block asks the TMA unit to bring the input of
// block b + D (b its own linear index) into L2 (bulk prefetches: no data
// reaches the SM and nothing waits on them), so that DRAM keeps streaming a
// later tile while this block transforms its own (passes B and D, always in
// FP32; the distance is in prefetch_distance).
//
// Block coordinates (x, y, z) of the block a.pf_ahead places after this one in
// launch order; false past the end of the grid.
template <typename T>
__device__ __forceinline__ bool grid_ahead(const PassArgs<T>& a, int& bx, int& by, int& bz) {
  const int64_t nblk = (int64_t)gridDim.x * gridDim.y * gridDim.z;
  const int64_t b = blockIdx.x + (int64_t)gridDim.x * (blockIdx.y + (int64_t)gridDim.y * blockIdx.z) + a.pf_ahead;
  if (b >= nblk) return false;
  bx = (int)(b % gridDim.x);
  const int64_t b1 = b / gridDim.x;
  by = (int)(b1 % gridDim.y);
  bz = (int)(b1 / gridDim.y);
  return true;
}
// Whether load case l still runs (its rows are worth prefetching).
template <typename T> __device__ __forceinline__ bool slot_runs(const PassArgs<T>& a, int l) {
  const CgState* cg = a.cg + l;
  return cg->active && !(a.cgphase && cg->status != ST_RUN);
}
// ---------------------------------------------------------------- pass A
// Resident blocks per SM the register budget is sized for.
template <typename T, int NT> __host__ __device__ constexpr int pass_a_min_blocks() {
  return sizeof(T) != 4 ? 1 : NT <= 384 ? 3 : NT <= 512 ? 2 : 1;
}

// grid (n_y/TY, n_z, L*G), G = 6 tetrahedra (6 components each) or 1 (nodal, 3).
// GS = 6 components per tetrahedron, or 3 for the nodal components (A_NODAL).
// NT is either the FFT's thread count or (tile variants 3, 4) the number of
// load units of the tile, so that every thread streams exactly one unit.
template <typename T, int NX, int TY, int NT, int GS>
__global__ void __launch_bounds__(NT, pass_a_min_blocks<T, NT>()) pass_a_3d(PassArgs<T> a) {
  using C = cplx<T>;
  constexpr int NP = TY / 2;
  constexpr int KX = NX / 2 + 1;
  constexpr int LD = ae_ld<NX>();
  extern __shared__ __align__(16) unsigned char smem_raw[];
  C* buf = reinterpret_cast<C*>(smem_raw);  // [GS][NP][LD]
  __shared__ double red[NT / 32];
  __shared__ T cols[NT];
  __shared__ int flag;
  constexpr bool nodal = GS == 3;
  const int G = nodal ? 1 : a.nq;
  const int l = blockIdx.z / G, grp = blockIdx.z % G;
  const int z = blockIdx.y, y0 = blockIdx.x * TY;
  const int ny = a.n[1], nz = a.n[2];
  CgState* cg = a.cg + l;
  pdl_begin();
  if (!cg->active) return;
  if (a.cgphase && cg->status != ST_RUN) return;
  const int c0 = nodal ? 0 : grp * 6;
  T beta = 0, alpha_prev = 0;
  bool use_old = false;
  if (a.amode == A_CG) { beta = cg_beta<T>(cg); alpha_prev = cg_alpha<T>(cg); use_old = cg->it > 0; }
  // two columns per unit: 6 components x 2 rows x (r, p, x) stay in registers
  const T acc = pass_a_load<T, NX, TY, GS, NT, LD, 2>(a, buf, l, c0, ((int64_t)z * ny + y0) * NX, nodal, beta,
                                                      alpha_prev, use_old);
  __syncthreads();
  smem_fft<T, NX, GS * NP, LD, NT, -1>(buf, a.tw[0]);
  pass_a_store<T, NX, TY, NT, LD>(buf, GS,
                                  a.spec + ((((int64_t)l * a.m + c0) * KX) * nz + z) * ny + y0,
                                  (int64_t)KX * nz * ny, (int64_t)nz * ny);

  if (a.amode == A_CG) {
    const double s = block_sum_cols<NT>(acc, cols);
    const int nblk = gridDim.x * gridDim.y * G;
    const int blk = blockIdx.x + gridDim.x * (blockIdx.y + gridDim.y * grp);
    double* part = a.part + (int64_t)l * a.part_stride;
    if (publish_partial(s, part, &cg->cnt_a, blk, nblk, &flag)) {
      const double pq = sum_partials<NT>(part, nblk, red);
      if (threadIdx.x == 0) finish_alpha(cg, pq);
    }
  }
}

// ---------------------------------------------------------------- pass B / D
// FFT along y.  grid (n_z/TZB, n_x/2+1, L*Cc).  FWD: spec1 pencils -> spec2
// chunks; !FWD: spec2 chunks -> spec1 pencils.
template <typename T, int NY, int TZB, int NT, bool FWD, int V = 0>
__global__ void __launch_bounds__(NT, sizeof(T) == 4 ? (NT <= 256 ? 4 : 2) : 1) pass_y_3d(PassArgs<T> a, int Cc) {
  using C = cplx<T>;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  constexpr int LD = FftSplit<NY, V>::LDO;  // odd: the chunk transposes are conflict-free
  C* buf = reinterpret_cast<C*>(smem_raw);  // [TZB][LD]
  const int l = blockIdx.z / Cc, c = blockIdx.z % Cc;
  const int kx = blockIdx.y, z0 = blockIdx.x * TZB;
  const int nz = a.n[2], KX = a.kx;
  CgState* cg = a.cg + l;
  pdl_begin();
  if (!cg->active) return;
  if (a.cgphase && cg->status != ST_RUN) return;
  const int64_t cbase = (((int64_t)l * a.m + c) * KX + kx);
  C* pencils = a.spec + (cbase * nz + z0) * NY;  // [zz][y], y contiguous
  C* chunks = a.spec2 + cbase * NY * nz + z0;     // [k_y][zz], zz contiguous
  // L2 prefetch of the later block's input (see grid_ahead): forward, its
  // TZB contiguous y-pencils (one request); inverse, its NY z-chunks of TZB
  // values
  int zb2, kx2, lc2;
  // the component that holds the second part of component i's nodal forces
  // (pair 1) or edge sums (pair 2: of x and y), less i; 0 where there is none
  auto second = [&](int i) -> int { return a.pair == 1 ? 3 : a.pair == 2 && i < 6 ? 9 : 0; };
  if (a.pf_ahead > 0 && grid_ahead(a, zb2, kx2, lc2) && slot_runs(a, lc2 / Cc)) {
    static_assert((TZB * sizeof(C)) % 16 == 0, "bulk prefetch sizes are multiples of 16 bytes");
    const int64_t cb2 = (((int64_t)(lc2 / Cc) * a.m + lc2 % Cc) * KX + kx2);
    const int z2 = zb2 * TZB;
    if (FWD) {
      const int s2 = second(lc2 % Cc);
      if (threadIdx.x < (s2 ? 2 : 1))
        prefetch_l2_bulk(a.spec + ((cb2 + s2 * (int64_t)threadIdx.x * KX) * nz + z2) * NY, (unsigned)(TZB * NY * sizeof(C)));
    } else {
      for (int k = threadIdx.x; k < NY; k += blockDim.x)
        prefetch_l2_bulk(a.spec2 + cb2 * NY * nz + z2 + (int64_t)k * nz, (unsigned)(TZB * sizeof(C)));
    }
  }
  if (FWD) {
    // step 1 reads whole y-pencils, step 2 writes z-chunks (zz fastest)
    auto st = [&](int zz, int k, C v) { chunks[(int64_t)k * nz + zz] = v; };
    if (a.resid) {
      // nodal state: this pass keeps the residual force R and transforms it (the
      // loads of several values come before their stores, which the compiler
      // could not reorder)
      const C* f1 = pencils + 3 * (int64_t)KX * nz * NY;
      C* res = pencils + 6 * (int64_t)KX * nz * NY;
      const bool upd = a.resid == 2;
      const T alpha = upd ? cg_alpha<T>(cg) : (T)1;
      constexpr int TOT = TZB * NY, U = 4;
      static_assert(TOT % NT == 0, "whole rounds");
      for (int i0 = threadIdx.x; i0 < TOT; i0 += U * NT) {
        C v[U], w[U], r[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
          const int i = i0 + u * NT;
          if (i < TOT) {
            v[u] = pencils[i];
            if (upd) { w[u] = f1[i]; r[u] = res[i]; }
          }
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
          const int i = i0 + u * NT;
          if (i < TOT) {
            if (upd) v[u] = csub(r[u], cscale(cadd(v[u], w[u]), alpha));
            else v[u] = cscale(v[u], (T)-1);
            res[i] = v[u];
            buf[(i / NY) * LD + i % NY] = v[u];
          }
        }
      }
      __syncthreads();
      auto ld = [&](int zz, int y) -> C { return buf[zz * LD + y]; };
      fft4<T, NY, TZB, LD, NT, -1, true, false, false, true, V>(buf, a.tw[1], ld, st);
    } else if (const int s2 = second(c)) {   // the two parts of the sums over elements (force_3d)
      const C* other = pencils + s2 * (int64_t)KX * nz * NY;
      auto ld = [&](int zz, int y) -> C {
        return cadd(pencils[(int64_t)zz * NY + y], other[(int64_t)zz * NY + y]);
      };
      fft4<T, NY, TZB, LD, NT, -1, false, false, false, true, V>(buf, a.tw[1], ld, st);
    } else {
      auto ld = [&](int zz, int y) -> C { return pencils[(int64_t)zz * NY + y]; };
      fft4<T, NY, TZB, LD, NT, -1, false, false, false, true, V>(buf, a.tw[1], ld, st);
    }
  } else {
    auto ld = [&](int zz, int k) -> C { return chunks[(int64_t)k * nz + zz]; };
    auto st = [&](int zz, int y, C v) { pencils[(int64_t)zz * NY + y] = v; };
    fft4<T, NY, TZB, LD, NT, +1, false, false, true, false, V>(buf, a.tw[1], ld, st);
  }
}

// ------------------------------------------------- pass B, finite elements
// From the x-transformed stresses of all 36 components, spec1 [c][k_x][z][y],
// the nodal forces t = B^H sigma and their y transform, spec2
// [j][k_x][k_y][z], j < 3.  A factor exp(-i k_a h_a) of B^H is a shift by one
// node along a, so B^H is applied here, where only x is transformed: every
// voxel gives the forces of its eight corners, the four with dx = 1 times
// exp(-i k_x h_x), and node (y, z) sums the corners (dy, dz) of voxels
// (y - dy, z - dz).  After this only the three nodal components are
// transformed along y and z, there and back, instead of all 36.  Bound by reading the
// 36-component spectrum once.
// A thread owns one y and marches in z over its lane's TZB / LN planes (one
// plane more on the low side), keeping the dz = 1 corners of the plane below in
// registers; the dy = 1 corners go to the neighbour row by a warp shuffle, and
// across warps through `edge`.  The loads of a plane's 36 components are
// independent, so a thread has up to 36 of them in flight.
// grid (n_z/TZB, n_x/2+1, L).
template <typename T, int NY, int TZB, int NT, int V>
__global__ void __launch_bounds__(NT, sizeof(T) == 4 ? (NT == 256 ? 2 : 6) : 1) pass_b_3d_fe(PassArgs<T> a) {
  using C = cplx<T>;
  constexpr int LN = NT / NY;            // z lanes
  constexpr int TZL = TZB / LN;          // planes per lane
  static_assert(NT % NY == 0 && TZB % LN == 0 && LN >= 1, "threads cover whole rows, lanes whole planes");
  constexpr int LD = FftSplit<NY, V>::LDO;
  constexpr int NW = NY > 32 ? NY / 32 : 1;   // warps per row
  extern __shared__ __align__(16) unsigned char smem_raw[];
  C* buf = reinterpret_cast<C*>(smem_raw);   // [3][TZB][LD]
  C* edge = buf + 3 * TZB * LD;              // [3][TZB][NW]: dy = 1 corners of each warp's last row
  const int l = blockIdx.z, kx = blockIdx.y, z0 = blockIdx.x * TZB;
  const int nz = a.n[2], KX = a.kx;
  CgState* cg = a.cg + l;
  pdl_begin();
  if (!cg->active) return;
  if (a.cgphase && cg->status != ST_RUN) return;
  const int y = threadIdx.x % NY, ln = threadIdx.x / NY;
  const int64_t cs = (int64_t)KX * nz * NY;  // component stride
  const C* src = a.spec + ((int64_t)l * a.m * KX + kx) * nz * NY + y;
  const C cex = cconj(a.ph[0][kx]);
  const C dx = cscale(csub(cex, mkc<T>(1, 0)), a.ih[0]);
  const C ey = cscale(cex, a.ih[1]), ez = cscale(cex, a.ih[2]);
  const T ihy = a.ih[1], ihz = a.ih[2], r2 = (T)kInvSqrt2;
  C c0[3], c1[3];   // dz = 1 corners of the plane below: (dy = 0, 1)
#pragma unroll
  for (int j = 0; j < 3; ++j) c0[j] = c1[j] = mkc<T>(0, 0);
  for (int zz = ln * TZL - 1; zz < (ln + 1) * TZL; ++zz) {
    const C* pl = src + (int64_t)((z0 + zz) & (nz - 1)) * NY;
    // d[dy + 2 dz][j]: corner forces of the voxel, the two dx corners combined
    C d[4][3];
#pragma unroll
    for (int k = 0; k < 4; ++k)
#pragma unroll
      for (int j = 0; j < 3; ++j) d[k][j] = mkc<T>(0, 0);
#pragma unroll
    for (int t = 0; t < 6; ++t) {
      C s[6];
#pragma unroll
      for (int c = 0; c < 6; ++c) s[c] = pl[(6 * t + c) * cs];
#pragma unroll
      for (int c = 3; c < 6; ++c) s[c] = cscale(s[c], r2);
      int at = 0;   // corner dx + 2 dy + 4 dz where the edge starts
#pragma unroll
      for (int e = 0; e < 3; ++e) {
        const int ax = kuhn_perm(t, e);
        const int lo = (at >> 1) & 3, hi = ((at | (1 << ax)) >> 1) & 3;
#pragma unroll
        for (int j = 0; j < 3; ++j) {
          const C sj = s[ax == j ? j : 6 - ax - j];   // sigma_ax,j: xx yy zz, yz xz xy
          if (ax == 0) {
            d[lo][j] = cadd(d[lo][j], cmul(dx, sj));
          } else {
            const C f = (at & 1) ? cmul(ax == 1 ? ey : ez, sj) : cscale(sj, ax == 1 ? ihy : ihz);
            d[lo][j] = csub(d[lo][j], f);
            d[hi][j] = cadd(d[hi][j], f);
          }
        }
        at |= 1 << ax;
      }
    }
    if (zz >= ln * TZL) {
#pragma unroll
      for (int j = 0; j < 3; ++j) {
        const C u = cadd(d[0][j], c0[j]), v = cadd(d[1][j], c1[j]);   // to nodes y and y + 1
        C vp;
        if constexpr (NY >= 32) {
          vp.x = __shfl_up_sync(0xffffffffu, v.x, 1);
          vp.y = __shfl_up_sync(0xffffffffu, v.y, 1);
          if ((threadIdx.x & 31) == 31) edge[(j * TZB + zz) * NW + y / 32] = v;
          if ((threadIdx.x & 31) == 0) vp = mkc<T>(0, 0);   // added from `edge` below
        } else {
          const int from = (threadIdx.x & 31 & ~(NY - 1)) | ((y + NY - 1) & (NY - 1));
          vp.x = __shfl_sync(0xffffffffu, v.x, from);
          vp.y = __shfl_sync(0xffffffffu, v.y, from);
        }
        buf[(j * TZB + zz) * LD + y] = cadd(u, vp);
      }
    }
#pragma unroll
    for (int j = 0; j < 3; ++j) { c0[j] = d[2][j]; c1[j] = d[3][j]; }
  }
  __syncthreads();
  if constexpr (NY >= 32) {
    for (int i = threadIdx.x; i < 3 * TZB * NW; i += NT) {
      const int row = i / NW, w = i % NW;
      C* p = buf + row * LD + 32 * w;
      *p = cadd(*p, edge[row * NW + (w + NW - 1) % NW]);
    }
    __syncthreads();
  }
  for (int j = 0; j < 3; ++j) {
    C* bj = buf + j * TZB * LD;
    C* chunks = a.spec2 + (((int64_t)l * a.m + j) * KX + kx) * NY * nz + z0;   // [k_y][zz], zz contiguous
    auto ld = [&](int zz, int yy) -> C { return bj[zz * LD + yy]; };
    auto st = [&](int zz, int k, C v) { chunks[(int64_t)k * nz + zz] = v; };
    fft4<T, NY, TZB, LD, NT, -1, true, false, false, true, V>(bj, a.tw[1], ld, st);
  }
}

// ---------------------------------------------------------------- pass C
// w^ = (B^H B)^-1 t^ at one wavevector (k != 0): column kz of the three
// component rows of buf, in place, scaled.
template <typename T, int LD>
__device__ __forceinline__ void solve_3d(cplx<T>* col, const cplx<T>* e, const T* ih, T scale) {
  using C = cplx<T>;
  C g[6][3];
  fe_gradients<T, 3>(e, ih, g);
  // M = B^H B = 1/2 sum_t (|g|^2 I + g g^H)
  T mdiag[3] = {0, 0, 0};
  C m01 = mkc<T>(0, 0), m02 = mkc<T>(0, 0), m12 = mkc<T>(0, 0);
#pragma unroll
  for (int t = 0; t < 6; ++t) {
    const T a0 = cabs2(g[t][0]), a1 = cabs2(g[t][1]), a2 = cabs2(g[t][2]);
    const T nn = a0 + a1 + a2;
    mdiag[0] += (T)0.5 * (nn + a0);
    mdiag[1] += (T)0.5 * (nn + a1);
    mdiag[2] += (T)0.5 * (nn + a2);
    m01 = cadd(m01, cscale(cmul(g[t][0], cconj(g[t][1])), (T)0.5));
    m02 = cadd(m02, cscale(cmul(g[t][0], cconj(g[t][2])), (T)0.5));
    m12 = cadd(m12, cscale(cmul(g[t][1], cconj(g[t][2])), (T)0.5));
  }
  const C t3[3] = {col[0], col[LD], col[2 * LD]};
  // w = M^-1 t by the adjugate of the Hermitian matrix
  // M = [[A, m01, m02], [conj m01, B, m12], [conj m02, conj m12, Cc]]
  const T A = mdiag[0], B = mdiag[1], Cc = mdiag[2];
  const T A00 = B * Cc - cabs2(m12);
  const T A11 = A * Cc - cabs2(m02);
  const T A22 = A * B - cabs2(m01);
  // adj[0][1] = m02 conj(m12) - m01 Cc ; adj[0][2] = m01 m12 - m02 B ; adj[1][2] = m02 conj(m01) - A m12
  const C A01 = csub(cmul(m02, cconj(m12)), cscale(m01, Cc));
  const C A02 = csub(cmul(m01, m12), cscale(m02, B));
  const C A12 = csub(cmul(m02, cconj(m01)), cscale(m12, A));
  const T det = A * A00 + (cmul(m01, cconj(A01))).x + (cmul(m02, cconj(A02))).x;
  const T id = scale / det;
  col[0] = cscale(cadd(cadd(cscale(t3[0], A00), cmul(A01, t3[1])), cmul(A02, t3[2])), id);
  col[LD] = cscale(cadd(cadd(cjmul(A01, t3[0]), cscale(t3[1], A11)), cmul(A12, t3[2])), id);
  col[2 * LD] = cscale(cadd(cadd(cjmul(A02, t3[0]), cjmul(A12, t3[1])), cscale(t3[2], A22)), id);
}

// Pass C of the finite elements: forward FFT along z, w^ = (B^H B)^-1 t^,
// inverse FFT, on the three nodal components; P pencils (k_x, k_y0 + i), i <
// P, per block.  Row b of the buffer is component b % 3 of pencil b / 3.  W =
// 9 (P = 1) reads the edge sums s_aj and writes the differences d_a w_j along
// the element edges as components 3 a + j (see pass_c_2d_fe).
// grid (n_x/2+1, n_y/P, L).
template <typename T, int NZ, int P, int NT, int V, int W>
__global__ void __launch_bounds__(NT, sizeof(T) == 8 ? 1 : W == 9 ? 8 : NT <= 384 ? 2 : 1) pass_c_3d_nodal(PassArgs<T> a) {
  using C = cplx<T>;
  constexpr int R = W * P;
  static_assert(W == 3 || (W == 9 && P == 1), "differences: one pencil per block");
  constexpr int LD = FftSplit<NZ, V>::LD;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  C* buf = reinterpret_cast<C*>(smem_raw);  // [W P][LD]
  __shared__ double red[NT / 32];
  __shared__ T cols[NT];
  __shared__ int flag;
  const int kx = blockIdx.x, ky0 = blockIdx.y * P, l = blockIdx.z;
  const int ny = a.n[1], KX = a.kx;
  CgState* cg = a.cg + l;
  pdl_begin();
  if (!cg->active) return;
  if (a.cgphase && cg->status != ST_RUN) return;
  const int64_t stride_c = (int64_t)KX * ny * NZ;
  C* base = a.spec2 + (int64_t)l * a.m * stride_c + ((int64_t)kx * ny + ky0) * NZ;
  auto ld_g = [&](int b, int z) -> C { return base[(b % W) * stride_c + (b / W) * NZ + z]; };
  auto st_s = [&](int b, int k, C v) { buf[b * LD + k] = v; };
  fft4<T, NZ, R, LD, NT, -1, false, true, false, false, V>(buf, a.tw[2], ld_g, st_s);
  Acc<T> acc;
  for (int i = threadIdx.x; i < P * NZ; i += NT) {
    const int pc = i / NZ, kz = i % NZ;
    C* col = buf + 3 * pc * LD + kz;
    if (kx == 0 && ky0 + pc == 0 && kz == 0) {
      // k = 0: the nodal solve has no mean (w^(0) = 0)
      for (int j = 0; j < W; ++j) col[j * LD] = mkc<T>(0, 0);
    } else {
      const C e[3] = {a.ph[0][kx], a.ph[1][ky0 + pc], a.ph[2][kz]};
      if constexpr (W == 9) {
#pragma unroll
        for (int j = 0; j < 3; ++j) {
          C t = mkc<T>(0, 0);
#pragma unroll
          for (int ax = 0; ax < 3; ++ax)
            t = cadd(t, cjmul(cscale(csub(e[ax], mkc<T>(1, 0)), a.ih[ax]), col[(3 * ax + j) * LD]));
          col[j * LD] = t;
        }
      }
      const C t[3] = {col[0], col[LD], col[2 * LD]};
      solve_3d<T, LD>(col, e, a.ih, a.inv_n);
      if (a.dot) {
        T d = 0;
#pragma unroll
        for (int j = 0; j < 3; ++j) d += t[j].x * col[j * LD].x + t[j].y * col[j * LD].y;
        acc.add(d);
      }
      if constexpr (W == 9) {
        const C w[3] = {col[0], col[LD], col[2 * LD]};
#pragma unroll
        for (int ax = 0; ax < 3; ++ax) {
          const C d = cscale(csub(e[ax], mkc<T>(1, 0)), a.ih[ax]);
#pragma unroll
          for (int j = 0; j < 3; ++j) col[(3 * ax + j) * LD] = cmul(d, w[j]);
        }
      }
    }
  }
  __syncthreads();
  auto ld_s = [&](int b, int z) -> C { return buf[b * LD + z]; };
  auto st_g = [&](int b, int k, C v) { base[(b % W) * stride_c + (b / W) * NZ + k] = v; };
  fft4<T, NZ, W * P, LD, NT, +1, true, false, false, false, V>(buf, a.tw[2], ld_s, st_g);
  if (a.dot) publish_rr<NT>(a, cg, acc, cols, red, &flag, kx == 0 || kx == KX - 1 ? 1.0 : 2.0, blockIdx.x + gridDim.x * blockIdx.y,
                            gridDim.x * gridDim.y, l);
}

// Pass C for one evaluation point per voxel (the derivatives of Secs. 2.3-2.5,
// m = 6): P = 6 pencils (k_x, k_y0 + i) of the 6 components per block, so
// that a block has the 36 transforms of the finite-element pass; row b is
// component b % 6 of pencil b / 6.  grid (n_x/2+1, ceil(n_y/P), L).
template <typename T, int NZ, int NT>
__global__ void __launch_bounds__(NT, sizeof(T) == 4 ? 2 : 1) pass_c_3d_q1(PassArgs<T> a) {
  using C = cplx<T>;
  constexpr int P = 6, R = 36;
  constexpr int LD = FftSplit<NZ>::LD;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  C* buf = reinterpret_cast<C*>(smem_raw);  // [R][LD]
  const int kx = blockIdx.x, ky0 = blockIdx.y * P, l = blockIdx.z;
  const int ny = a.n[1], KX = a.kx;
  CgState* cg = a.cg + l;
  pdl_begin();
  if (!cg->active) return;
  if (a.cgphase && cg->status != ST_RUN) return;
  const int64_t stride_c = (int64_t)KX * ny * NZ;
  C* base = a.spec2 + (int64_t)l * a.m * stride_c + ((int64_t)kx * ny + ky0) * NZ;
  auto ld_g = [&](int b, int z) -> C {
    return (ky0 + b / 6 < ny) ? base[(b % 6) * stride_c + (b / 6) * NZ + z] : mkc<T>(0, 0);
  };
  auto st_s = [&](int b, int k, C v) { buf[b * LD + k] = v; };
  fft4<T, NZ, R, LD, NT, -1, false, true, false, false>(buf, a.tw[2], ld_g, st_s);
  for (int i = threadIdx.x; i < P * NZ; i += NT) {
    const int pc = i / NZ, kz = i % NZ, ky = ky0 + pc;
    if (ky >= ny) continue;
    C sv[6];
#pragma unroll
    for (int c = 0; c < 6; ++c) sv[c] = buf[(6 * pc + c) * LD + kz];
    if (kx == 0 && ky == 0 && kz == 0) {
#pragma unroll
      for (int c = 0; c < 6; ++c) sv[c] = mkc<T>(0, 0);
    } else {
      const int j[3] = {kx, ky, kz};
      const C e[3] = {a.ph[0][kx], a.ph[1][ky], a.ph[2][kz]};
      C g[2][3];
      const int nq = deriv_symbols<T, 3>(a.deriv, j, a.n, e, a.ih, g);
      project_generic<T, 3>(sv, g, nq, a.inv_n);
    }
#pragma unroll
    for (int c = 0; c < 6; ++c) buf[(6 * pc + c) * LD + kz] = sv[c];
  }
  __syncthreads();
  auto ld_s = [&](int b, int z) -> C { return buf[b * LD + z]; };
  auto st_g = [&](int b, int k, C v) {
    if (ky0 + b / 6 < ny) base[(b % 6) * stride_c + (b / 6) * NZ + k] = v;
  };
  fft4<T, NZ, R, LD, NT, +1, true, false, false, false>(buf, a.tw[2], ld_s, st_g);
}

// Pass C for finite strain (P_FINITE): one (k_x, k_y) pencil of the 54
// deformation-gradient components (6 tetrahedra x 3 x 3) per block.
// grid (n_x/2+1, n_y, L).
template <typename T, int NZ, int NT>
__global__ void __launch_bounds__(NT, 1) pass_c_3d_fs(PassArgs<T> a) {
  using C = cplx<T>;
  constexpr int R = 54;
  constexpr int LD = FftSplit<NZ>::LD;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  C* buf = reinterpret_cast<C*>(smem_raw);  // [R][LD]
  const int kx = blockIdx.x, ky = blockIdx.y, l = blockIdx.z;
  const int ny = a.n[1], KX = a.kx;
  CgState* cg = a.cg + l;
  pdl_begin();
  if (!cg->active) return;
  if (a.cgphase && cg->status != ST_RUN) return;
  const int64_t stride_c = (int64_t)KX * ny * NZ;
  C* pen = a.spec2 + (int64_t)l * a.m * stride_c + ((int64_t)kx * ny + ky) * NZ;
  auto ld_g = [&](int c, int z) -> C { return pen[c * stride_c + z]; };
  auto st_s = [&](int c, int k, C v) { buf[c * LD + k] = v; };
  fft4<T, NZ, R, LD, NT, -1, false, true, false, false>(buf, a.tw[2], ld_g, st_s);
  for (int kz = threadIdx.x; kz < NZ; kz += NT) {
    const C e[3] = {a.ph[0][kx], a.ph[1][ky], a.ph[2][kz]};
    C g[6][3];
    fe_gradients<T, 3>(e, a.ih, g);
    auto col = [&](int c) -> C& { return buf[c * LD + kz]; };
    project_finite<T, 3, 6>(col, g, a.inv_n, kx == 0 && ky == 0 && kz == 0);
  }
  __syncthreads();
  auto ld_s = [&](int c, int z) -> C { return buf[c * LD + z]; };
  auto st_g = [&](int c, int k, C v) { pen[c * stride_c + k] = v; };
  fft4<T, NZ, R, LD, NT, +1, true, false, false, false>(buf, a.tw[2], ld_s, st_g);
}

// ---------------------------------------------------------------- pass E
// grid (n_y/TY, n_z, L*G): G = 6 tetrahedra (6 components each) or one group
// of the 3 nodal components (E_NODAL); inverse real FFT along x and update.
template <typename T, int NX, int TY, int NT, int GE>
__global__ void __launch_bounds__(NT, (sizeof(T) == 4 && NT <= 384) ? 3 : 1) pass_e_3d(PassArgs<T> a) {
  using C = cplx<T>;
  constexpr int NP = TY / 2;
  constexpr int KX = NX / 2 + 1;
  constexpr int LD = ae_ld<NX>();
  extern __shared__ __align__(16) unsigned char smem_raw[];
  C* buf = reinterpret_cast<C*>(smem_raw);  // [GE][NP][LD]
  __shared__ double red[NT / 32];
  __shared__ T cols[NT];
  __shared__ int flag;
  constexpr bool nodal = GE == 3;
  const int G = nodal ? 1 : a.nq;
  const int l = blockIdx.z / G, grp = blockIdx.z % G;
  const int z = blockIdx.y, y0 = blockIdx.x * TY;
  const int ny = a.n[1], nz = a.n[2];
  const int64_t N = a.N;
  CgState* cg = a.cg + l;
  pdl_begin();
  if (!cg->active) return;
  if (a.cgphase && cg->status != ST_RUN) return;
  const int c0 = nodal ? 0 : grp * GE;
  pass_e_unpack<T, NX, TY, NT, LD>(buf, a.spec + ((((int64_t)l * a.m + c0) * KX) * nz + z) * ny, GE,
                                   (int64_t)KX * nz * ny, (int64_t)nz * ny, y0, ny - 1);
  __syncthreads();
  T acc = 0;
  const T alpha = (a.emode == E_CG) ? cg_alpha<T>(cg) : (T)0;
  auto ld_s = [&](int b, int x) -> C { return buf[b * LD + x]; };
  PassEStore<T, NX, NP> st{&a, GE, ((int64_t)z * ny + y0) * NX, ((int64_t)l * a.m + c0) * N, (int64_t)l * 3 * N,
                           alpha, &acc};
  fft4<T, NX, GE * NP, LD, NT, +1, true, false, false, false, 0, decltype(ld_s), decltype(st), true>(buf, a.tw[0],
                                                                                                  ld_s, st);

  if (a.emode == E_CG || a.emode == E_INIT) {
    const double s = block_sum_cols<NT>(acc, cols);
    const int nblk = gridDim.x * gridDim.y * G;
    const int blk = blockIdx.x + gridDim.x * (blockIdx.y + gridDim.y * grp);
    double* part = a.part + (int64_t)l * a.part_stride;
    if (publish_partial(s, part, &cg->cnt_e, blk, nblk, &flag)) {
      const double rr = sum_partials<NT>(part, nblk, red);
      if (threadIdx.x == 0) finish_rr(cg, rr, a.emode == E_INIT);
    }
  }
}

// Last pass of the finite elements: from w(k_x, z, y) of the three nodal
// components (pass D) the inverse x FFT of TY + 1 rows of planes z and z + 1,
// then in real space the strains q = B w of the six tetrahedra of every voxel of
// the TY rows and the update of all 36 components.  Transforming w needs 3 TY + 4
// transforms where the components need 18 TY, and reads 1/12 of the spectrum;
// what is left is the r traffic (read and written once), which bounds it.
// Two real rows share a complex transform: w_0 and w_1 of a row, and w_2 of rows
// 2 i and 2 i + 1.  Every node's values then come from the same transforms in
// all blocks that use them (a tile's last row is the next one's first, plane z +
// 1 is the next block's plane z), and q is the strain of one nodal field.
// Pairing planes z and z + 1 (3 TY + 3 transforms) rounds a node's values
// differently in the two blocks: the differences of that are no strain field, CG
// cannot remove them from r, and on flat voxels (1 : 1000, FP32) it did not
// converge.
// W = 9: the spectrum holds the edge differences of w instead (see
// pass_c_2d_fe); plane z in the real, plane z + 1 in the imaginary part.
// grid (n_y/TY, n_z, L).
// In FP32 the r loads of the update go through a ring of the thread's own
// shared-memory slots (cp.async, six tetrahedra deep): issued before the
// spectrum is unpacked, they keep DRAM busy during the transforms, and in the
// update no store waits for the loads behind it (us per iteration, without and
// with, taken with the planes paired: 256 x 256 x 64 309, 289; 128^3 156, 149;
// 64^3, six load cases 147, 114.  Paired within a plane: 297, 154, 115).
template <typename T, int NT, int W> __host__ __device__ constexpr bool e_fe_ring() {
  return sizeof(T) == 4 && W == 3 && NT <= 256;   // else it does not fit beside the rows
}
template <int W, int TY> __host__ __device__ constexpr int e_fe_rows() { return W == 3 ? 3 * TY + 4 : W * (TY + 1); }
template <int NX> __host__ __device__ constexpr int e_fe_ld() {
  // 9 (mod 16): the TY + 1 rows that consecutive lanes unpack at one column
  // fall on different banks
  return FftSplit<NX>::LD + ((9 - FftSplit<NX>::LD % 16) + 16) % 16;
}
template <typename T, int NX, int TY, int NT, int MB, int W>
__global__ void __launch_bounds__(NT, MB) pass_e_3d_fe(PassArgs<T> a) {
  using C = cplx<T>;
  constexpr int KX = NX / 2 + 1;
  constexpr int NR = TY + 1;
  constexpr int NP = TY / 2 + 1;   // row pairs of w_2
  constexpr int R = e_fe_rows<W, TY>();
  static_assert(W == 9 || R == 2 * (NR + NP), "rows of the two planes");
  constexpr int LD = e_fe_ld<NX>();
  extern __shared__ __align__(16) unsigned char smem_raw[];
  C* buf = reinterpret_cast<C*>(smem_raw);  // W = 3: [2][NR] rows (w_0, w_1), [2][NP] pairs of w_2; 9: [W][NR]
  __shared__ double red[NT / 32];
  __shared__ T cols[sizeof(T) == 4 ? NT / 16 : NT];   // (1 KB less holds a fourth block at n_x = 128)
  __shared__ int flag;
  const int l = blockIdx.z, z = blockIdx.y, y0 = blockIdx.x * TY;
  const int ny = a.n[1], nz = a.n[2];
  const int64_t N = a.N;
  CgState* cg = a.cg + l;
  pdl_begin();
  if (!cg->active) return;
  if (a.cgphase && cg->status != ST_RUN) return;
  const bool cgm = a.emode == E_CG;
  const int64_t vox0 = (int64_t)l * a.m * N + ((int64_t)z * ny + y0) * NX;
  // the r values of this thread's next six tetrahedra, copied into its own
  // slots while the spectrum is unpacked and transformed (see e_fe_ring)
  constexpr bool RING = e_fe_ring<T, NT, W>();
  constexpr int VL = (RING && NX >= 256) ? 2 : 1; // voxels of a thread's unit (256: 298 -> 289 us; 64^3: 114, 130 with 2)
  constexpr int UNITS = TY * (NX / VL);
  T* ring = reinterpret_cast<T*>(buf + R * LD);   // [6][6][NT] units
  auto issue = [&](int i, int t) {
    if (cgm && i < UNITS) {
      const T* src = a.r + vox0 + VL * i;
#pragma unroll
      for (int s = 0; s < 6; ++s)
        copy_async<VL * (int)sizeof(T)>(ring + ((6 * t + s) * NT + threadIdx.x) * VL, src + (6 * t + s) * N);
    }
    copy_async_commit();
  };
  if constexpr (RING) {
#pragma unroll
    for (int t = 0; t < 6; ++t) issue(threadIdx.x, t);
  }
  {
    const C* pa = a.spec + ((int64_t)l * a.m * KX * nz + z) * ny;
    const C* pb = a.spec + ((int64_t)l * a.m * KX * nz + ((z + 1) & (nz - 1))) * ny;
    const int64_t cs = (int64_t)KX * nz * ny;
    auto pack = [&](C* row, int k, C va, C vb) {
      if (k == 0 || k == NX / 2) { va.y = 0; vb.y = 0; }  // C2R ignores these imaginary parts
      row[k] = mkc<T>(va.x - vb.y, va.y + vb.x);                                  // X_a + i X_b
      if (k > 0 && k < NX / 2) row[NX - k] = mkc<T>(va.x + vb.y, vb.x - va.y);    // conj(X_a) + i conj(X_b)
    };
    // items i -> (row b of NB rows a plane or component, k_x, plane or component p),
    // loaded UB at a time
    constexpr int UB = 4;
    auto unpack = [&](auto nb, int np, C* dst, auto&& load) {
      constexpr int NB = decltype(nb)::value;
      const int tot = np * KX * NB;
      for (int i0 = threadIdx.x; i0 < tot; i0 += UB * NT) {
        C v[UB][2];
#pragma unroll
        for (int u = 0; u < UB; ++u) {
          const int i = i0 + u * NT;
          if (i < tot) load(v[u], i % NB, (i / NB) % KX, i / (NB * KX));
        }
#pragma unroll
        for (int u = 0; u < UB; ++u) {
          const int i = i0 + u * NT;
          if (i < tot) pack(dst + ((i / (NB * KX)) * NB + i % NB) * LD, (i / NB) % KX, v[u][0], v[u][1]);
        }
      }
    };
    if constexpr (W == 3) {
      unpack(std::integral_constant<int, NR>{}, 2, buf, [&](C* v, int y, int k, int p) {
        const C* s = (p ? pb : pa) + (int64_t)k * nz * ny + ((y0 + y) & (ny - 1));
        v[0] = s[0];
        v[1] = s[cs];
      });
      unpack(std::integral_constant<int, NP>{}, 2, buf + 2 * NR * LD, [&](C* v, int pr, int k, int p) {
        cload2<T>(v, (p ? pb : pa) + 2 * cs + (int64_t)k * nz * ny + ((y0 + 2 * pr) & (ny - 1)));
      });
    } else {
      unpack(std::integral_constant<int, NR>{}, W, buf, [&](C* v, int y, int k, int j) {
        const int64_t o = j * cs + (int64_t)k * nz * ny + ((y0 + y) & (ny - 1));
        v[0] = pa[o];
        v[1] = pb[o];
      });
    }
  }
  __syncthreads();
  smem_fft<T, NX, R, LD, NT, +1>(buf, a.tw[0]);
  const T alpha = cgm ? cg_alpha<T>(cg) : (T)0;
  const T ih[3] = {a.ih[0], a.ih[1], a.ih[2]};
  const T r2 = (T)kInvSqrt2;
  Acc<T> acc;
  for (int i = threadIdx.x; i < UNITS; i += NT) {
    const int yy = i / (NX / VL), x = (i % (NX / VL)) * VL;
    const int64_t v0 = vox0 + (int64_t)yy * NX + x;
    // node values at (x + q, y + dy), planes z and z + 1
    constexpr int NV = W == 3 ? 2 : W;
    C n[NV][2][VL + 1];         // W = 3: [dz] (w_0, w_1); 9: [component] (z, z + 1)
    T n2[2][2][VL + 1];         // W = 3: w_2, [dz]
#pragma unroll
    for (int j = 0; j < NV; ++j)
#pragma unroll
      for (int dy = 0; dy < 2; ++dy)
#pragma unroll
        for (int q = 0; q <= VL; ++q) {
          const int xq = (x + q) & (NX - 1);
          n[j][dy][q] = buf[(j * NR + yy + dy) * LD + xq];
          if constexpr (W == 3) {
            const C* w = buf + (2 * NR + j * NP + (yy + dy) / 2) * LD + xq;
            n2[j][dy][q] = ((yy + dy) & 1) ? w->y : w->x;
          }
        }
    auto corner = [&](int c, int j, int q) -> T {   // corner c = dx + 2 dy + 4 dz of voxel x + q
      const int dx = c & 1, dy = (c >> 1) & 1, dz = (c >> 2) & 1;
      if constexpr (W == 3) return j == 0 ? n[dz][dy][q + dx].x : j == 1 ? n[dz][dy][q + dx].y : n2[dz][dy][q + dx];
      else return dz ? n[j][dy][q + dx].y : n[j][dy][q + dx].x;
    };
    T vs = 0;
#pragma unroll
    for (int t = 0; t < 6; ++t) {
      T rv[6][VL];
      if (cgm) {
        if constexpr (RING) copy_async_wait<5>();
#pragma unroll
        for (int s = 0; s < 6; ++s)
          vloadn<T, VL>(rv[s], RING ? ring + ((6 * t + s) * NT + threadIdx.x) * VL : a.r + v0 + (6 * t + s) * N);
      }
      if constexpr (RING) issue(i + NT, t);
      const int ax[3] = {kuhn_perm(t, 0), kuhn_perm(t, 1), kuhn_perm(t, 2)};
      const int v1 = 1 << ax[0], v2 = v1 | (1 << ax[1]);
      const int at[4] = {0, v1, v2, 7};
      T q[6][VL];
#pragma unroll
      for (int k = 0; k < VL; ++k) {
        T H[3][3];   // H[a][j] = d w_j / d x_a
#pragma unroll
        for (int e = 0; e < 3; ++e)
#pragma unroll
          for (int j = 0; j < 3; ++j)
            H[ax[e]][j] = W == 9 ? corner(at[e], 3 * ax[e] + j, k)
                                 : (corner(at[e + 1], j, k) - corner(at[e], j, k)) * ih[ax[e]];
        q[0][k] = H[0][0]; q[1][k] = H[1][1]; q[2][k] = H[2][2];
        q[3][k] = r2 * (H[1][2] + H[2][1]);
        q[4][k] = r2 * (H[0][2] + H[2][0]);
        q[5][k] = r2 * (H[0][1] + H[1][0]);
      }
#pragma unroll
      for (int s = 0; s < 6; ++s) vs += strain_update<T, VL>(a, v0 + (6 * t + s) * N, rv[s], q[s], alpha);
    }
    acc.add(vs);
  }
  if (cgm || a.emode == E_INIT) {
    const double s = block_sum_acc<NT>(acc, cols);
    const int nblk = gridDim.x * gridDim.y, blk = blockIdx.x + gridDim.x * blockIdx.y;
    double* part = a.part + (int64_t)l * a.part_stride;
    if (publish_partial(s, part, &cg->cnt_e, blk, nblk, &flag)) {
      const double rr = sum_partials<NT>(part, nblk, red);
      if (threadIdx.x == 0) finish_rr(cg, rr, a.emode == E_INIT);
    }
  }
}

// ------------------------------------------------------------ launchers
template <typename T> struct Tile3D;
template <> struct Tile3D<float> { static constexpr int TY = 8; static constexpr int TZB = 16; };
template <> struct Tile3D<double> { static constexpr int TY = 4; static constexpr int TZB = 8; };

template <typename T> constexpr int tile_rows3(int v) {
  return v == 1 ? Tile3D<T>::TY / 2 : v == 2 ? Tile3D<T>::TY * 2 : Tile3D<T>::TY;
}

// Load units of a pass A tile (see pass_a_load: two rows x one 16-byte vector
// of every component of one half of an element).
template <typename T, int NX, int TY> constexpr int pass_a_units3() { return 2 * (TY / 2) * (NX / Vec16<T>::n); }
template <int A, int B> constexpr int max_i() { return A > B ? A : B; }

// Prefetch distance (blocks ahead, see grid_ahead): the blocks resident at once
// (occ per SM x SMs) divided by div.  What pays is about 4 to 10 MB of
// prefetched rows in flight.  Measured at 256^3 with all 36 components (FP32,
// ms per CG iteration):
//   pass B (32 KB per block): 0.86 without, 0.81 / 0.77 / 0.72 / 0.69 / 0.72
//     at div 16 / 8 / 4 / 2 / 1;
//   pass D (32 KB per block, scattered z-chunks): 0.85 without, 0.83 / 0.82 /
//     0.82 / 0.82 / 0.84.
inline int prefetch_distance(int occ, int div) {
  const int d = occ * device_sm_count() / div;
  return d > 1 ? d : 1;
}

template <typename T, int NX, int TY, bool BY_UNITS = false, int GS = 6>
cudaError_t launch_a_3d_t(const PassArgs<T>& a, cudaStream_t s) {
  constexpr int NF = fft_threads<NX, GS * (TY / 2)>();
  constexpr int NU = (pass_a_units3<T, NX, TY>() + 31) / 32 * 32;
  constexpr int NT = BY_UNITS ? (max_i<NF, NU>() > 1024 ? NF : max_i<NF, NU>()) : NF;
  const size_t sm = sizeof(cplx<T>) * GS * (TY / 2) * ae_ld<NX>();
  auto k = pass_a_3d<T, NX, TY, NT, GS>;
  static DeviceOnce attr;
  attr.run(current_device(), [&] { set_smem_attrs(k, sm); });
  dim3 grid(a.n[1] / TY, a.n[2], a.L * (GS == 3 ? 1 : a.nq));
  return launch_pass(a.pdl, k, grid, NT, sm, s, a);
}
template <typename T, int NX, int TY, int GE = 6>
cudaError_t launch_e_3d_t(const PassArgs<T>& a, cudaStream_t s) {
  constexpr int NT = fft_threads<NX, GE * (TY / 2)>();
  const size_t sm = sizeof(cplx<T>) * GE * (TY / 2) * ae_ld<NX>();
  auto k = pass_e_3d<T, NX, TY, NT, GE>;
  static DeviceOnce attr;
  attr.run(current_device(), [&] { set_smem_attrs(k, sm); });
  dim3 grid(a.n[1] / TY, a.n[2], a.L * (GE == 3 ? 1 : a.nq));
  return launch_pass(a.pdl, k, grid, NT, sm, s, a);
}
template <typename T, int NX, int TY, int W = 3>
cudaError_t launch_e_3d_fe_t(const PassArgs<T>& a, cudaStream_t s) {
  constexpr int R = e_fe_rows<W, TY>();
  constexpr int NT = fft_threads<NX, R>();
  constexpr size_t sm = sizeof(cplx<T>) * R * e_fe_ld<NX>() + (e_fe_ring<T, NT, W>() ? sizeof(T) * 36 * (NX >= 256 ? 2 : 1) * NT : 0);
  constexpr int MB = sizeof(T) == 8 ? 1 : W == 9 ? (NT <= 448 ? 2 : 1) : NT <= 256 ? (NX >= 256 ? 2 : 4) : NT <= 448 ? 2 : 1;
  auto k = pass_e_3d_fe<T, NX, TY, NT, MB, W>;
  static DeviceOnce attr;
  attr.run(current_device(), [&] { set_smem_attrs(k, sm); });
  return launch_pass(a.pdl, k, dim3(a.n[1] / TY, a.n[2], a.L), NT, sm, s, a);
}
// Tile variants of pass A on all components: 0 default rows per block, 1 half,
// 2 double (threads = the FFT's); 3 default rows and 4 half rows with one
// thread per load unit (FP64: the derivatives without a finite-element stencil,
// and finite strain); 5 (FP32, n_x >= 128, CG iterations) the pipelined
// persistent pass with bulk-copied rows (pass3d_pipe.cuh), which uses variant 0
// for more load cases than it keeps sums for.
template <typename T, int NX>
cudaError_t launch_a_3d_n(const PassArgs<T>& a, cudaStream_t s) {
  // the three nodal components: twice the rows, so that a block holds as many
  // transforms as with six components (256^3, FP32: 137 us with the six-component
  // tile, half of whose transforms were padding)
  if (a.amode == A_NODAL) return launch_a_3d_t<T, NX, tile_rows3<T>(2), false, 3>(a, s);
  if constexpr (sizeof(T) == 4 && NX >= 128) {
    if (a.var_a == 5 && a.amode == A_CG && a.L <= kPipeMaxL && a.n[1] >= 4) return launch_a_3d_pipe<NX>(a, s);
  }
  if constexpr (NX >= 64 && sizeof(T) == 8) {
    if (a.var_a == 1) return launch_a_3d_t<T, NX, tile_rows3<T>(1)>(a, s);
    if (a.var_a == 2 && a.n[1] >= tile_rows3<T>(2)) return launch_a_3d_t<T, NX, tile_rows3<T>(2)>(a, s);
    if (a.var_a == 3) return launch_a_3d_t<T, NX, tile_rows3<T>(0), true>(a, s);
    if (a.var_a == 4) return launch_a_3d_t<T, NX, tile_rows3<T>(1), true>(a, s);
  }
  return launch_a_3d_t<T, NX, tile_rows3<T>(0)>(a, s);
}
// Tile variants of pass E: 0 default rows per block, 1 half, 2 double; with
// n_x >= 128 in FP32 also 3 and 4, the same tiles as 0 and 1.
template <typename T, int NX>
cudaError_t launch_e_3d_n(const PassArgs<T>& a, cudaStream_t s) {
  if (fe_path(a) && (a.emode == E_CG || a.emode == E_INIT || a.emode == E_OUT)) {
    if (a.grads) return launch_e_3d_fe_t<T, NX, tile_rows3<T>(1), 9>(a, s);
    if constexpr (NX >= 64) {
      if (a.var_e == 1 || a.var_e == 4) return launch_e_3d_fe_t<T, NX, tile_rows3<T>(1)>(a, s);
      if (a.var_e == 2 && a.n[1] >= tile_rows3<T>(2)) return launch_e_3d_fe_t<T, NX, tile_rows3<T>(2)>(a, s);
    }
    return launch_e_3d_fe_t<T, NX, tile_rows3<T>(0)>(a, s);
  }
  // the three nodal components: twice the rows, as in pass A
  if (a.emode == E_NODAL || a.emode == E_NOUT) return launch_e_3d_t<T, NX, tile_rows3<T>(2), 3>(a, s);
  if constexpr (sizeof(T) == 4) return cudaErrorInvalidValue;   // all components: FP64 only
  else {
    if constexpr (NX >= 64) {
      if (a.var_e == 1) return launch_e_3d_t<T, NX, tile_rows3<T>(1)>(a, s);
      if (a.var_e == 2 && a.n[1] >= tile_rows3<T>(2)) return launch_e_3d_t<T, NX, tile_rows3<T>(2)>(a, s);
    }
    return launch_e_3d_t<T, NX, tile_rows3<T>(0)>(a, s);
  }
}
template <typename T, int NY, bool FWD, int V>
cudaError_t launch_y_3d_v(const PassArgs<T>& a, cudaStream_t s) {
  constexpr int TZB = Tile3D<T>::TZB;
  constexpr int NT = fft_threads<NY, TZB, V>();
  const size_t sm = sizeof(cplx<T>) * TZB * FftSplit<NY, V>::LDO;
  auto k = pass_y_3d<T, NY, TZB, NT, FWD, V>;
  static DeviceOnce attr;
  static int occ[kMaxDevices] = {0};
  const int dev = current_device();
  attr.run(dev, [&] {
    set_smem_attrs(k, sm);
    if (dev >= 0 && dev < kMaxDevices) cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ[dev], k, NT, sm);
  });
  const int Cc = !fe_path(a) ? a.m : a.grads ? 9 : 3;   // finite elements: edge sums and differences, or t and w
  dim3 grid(a.n[2] / TZB, a.kx, a.L * Cc);
  if (sizeof(T) == 4) {
    PassArgs<T> b = a;
    b.pf_ahead = prefetch_distance((dev >= 0 && dev < kMaxDevices) ? occ[dev] : 0, 2);
    return launch_pass(b.pdl, k, grid, NT, sm, s, b, Cc);
  } else {
    return launch_pass(a.pdl, k, grid, NT, sm, s, a, Cc);
  }
}
// Pass B of the finite elements from all components (forward).
template <typename T, int NY, int V>
cudaError_t launch_b_3d_fe(const PassArgs<T>& a, cudaStream_t s) {
  constexpr int TZB = Tile3D<T>::TZB;
  constexpr int NT = NY >= 128 ? NY : 128;
  constexpr size_t sm = sizeof(cplx<T>) * (3 * TZB * FftSplit<NY, V>::LDO + 3 * TZB * (NY > 32 ? NY / 32 : 1));
  auto k = pass_b_3d_fe<T, NY, TZB, NT, V>;
  static DeviceOnce attr;
  attr.run(current_device(), [&] { set_smem_attrs(k, sm); });
  return launch_pass(a.pdl, k, dim3(a.n[2] / TZB, a.kx, a.L), NT, sm, s, a);
}
// Split variant of the y transforms (passes B and D): a.var_y.
template <typename T, int NY, bool FWD>
cudaError_t launch_y_3d_n(const PassArgs<T>& a, cudaStream_t s) {
  if constexpr (FWD && sizeof(T) == 4) {   // after the pipelined first pass (tile variant 5, FP32)
    if (fe_path(a) && !a.pair && a.pmode != P_NODAL_IN && a.pmode != P_SOLVE) {
      if constexpr (fft_split_count<NY>() > 1) {
        if (a.var_y == 1) return launch_b_3d_fe<T, NY, 1>(a, s);
      }
      return launch_b_3d_fe<T, NY, 0>(a, s);
    }
  }
  if constexpr (fft_split_count<NY>() > 1) {
    if (a.var_y == 1) return launch_y_3d_v<T, NY, FWD, 1>(a, s);
  }
  return launch_y_3d_v<T, NY, FWD, 0>(a, s);
}
template <typename T, int NY> cudaError_t launch_yf_3d_n(const PassArgs<T>& a, cudaStream_t s) {
  return launch_y_3d_n<T, NY, true>(a, s);
}
template <typename T, int NY> cudaError_t launch_yb_3d_n(const PassArgs<T>& a, cudaStream_t s) {
  return launch_y_3d_n<T, NY, false>(a, s);
}
// Pass C of the finite elements with split variant V (a.var_c): 8 pencils per
// block (n_y >= 16).
template <typename T, int NZ, int V, int W = 3>
cudaError_t launch_c_3d_v(const PassArgs<T>& a, cudaStream_t s) {
  constexpr int P = W == 9 ? 1 : 8;
  constexpr int NT = fft_threads<NZ, W * P, V>();
  const size_t sm = sizeof(cplx<T>) * W * P * FftSplit<NZ, V>::LD;
  auto k = pass_c_3d_nodal<T, NZ, P, NT, V, W>;
  static DeviceOnce attr;
  attr.run(current_device(), [&] { set_smem_attrs(k, sm); });
  return launch_pass(a.pdl, k, dim3(a.kx, a.n[1] / P, a.L), NT, sm, s, a);
}

template <typename T, int NZ>
cudaError_t launch_c_3d_n(const PassArgs<T>& a, cudaStream_t s) {
  if constexpr (sizeof(T) == 8) {   // all components: FP64 only
    if (a.pmode == P_FINITE) {
      constexpr int NTf = fft_threads<NZ, 54>();
      const size_t smf = sizeof(cplx<T>) * 54 * FftSplit<NZ>::LD;
      if (smf > 227 * 1024) return cudaErrorInvalidConfiguration;   // FP64 at n_z = 256
      auto kf = pass_c_3d_fs<T, NZ, NTf>;
      static DeviceOnce attrf;
      attrf.run(current_device(), [&] { set_smem_attrs(kf, smf); });
      return launch_pass(a.pdl, kf, dim3(a.kx, a.n[1], a.L), NTf, smf, s, a);
    }
    if (!fe_path(a)) {
      constexpr int NT1 = fft_threads<NZ, 36>();
      const size_t sm1 = sizeof(cplx<T>) * 36 * FftSplit<NZ>::LD;
      auto k1 = pass_c_3d_q1<T, NZ, NT1>;
      static DeviceOnce attr1;
      attr1.run(current_device(), [&] { set_smem_attrs(k1, sm1); });
      return launch_pass(a.pdl, k1, dim3(a.kx, (a.n[1] + 5) / 6, a.L), NT1, sm1, s, a);
    }
  }
  if constexpr (fft_split_count<NZ>() > 1) {
    if (a.var_c == 1) return a.grads ? launch_c_3d_v<T, NZ, 1, 9>(a, s) : launch_c_3d_v<T, NZ, 1>(a, s);
  }
  return a.grads ? launch_c_3d_v<T, NZ, 0, 9>(a, s) : launch_c_3d_v<T, NZ, 0>(a, s);
}

#define RVE_DISPATCH_N3(nval, FN, ...)                     \
  switch (nval) {                                          \
    case 16: return FN<T, 16>(__VA_ARGS__);                \
    case 32: return FN<T, 32>(__VA_ARGS__);                \
    case 64: return FN<T, 64>(__VA_ARGS__);                \
    case 128: return FN<T, 128>(__VA_ARGS__);              \
    case 256: return FN<T, 256>(__VA_ARGS__);              \
    default: return cudaErrorInvalidValue;                 \
  }

template <typename T> cudaError_t launch_pass_a_3d(const PassArgs<T>& a, cudaStream_t s) {
  RVE_DISPATCH_N3(a.n[0], launch_a_3d_n, a, s)
}
template <typename T> cudaError_t launch_pass_b_3d(const PassArgs<T>& a, cudaStream_t s) {
  RVE_DISPATCH_N3(a.n[1], launch_yf_3d_n, a, s)
}
template <typename T> cudaError_t launch_pass_c_3d(const PassArgs<T>& a, cudaStream_t s) {
  RVE_DISPATCH_N3(a.n[2], launch_c_3d_n, a, s)
}
template <typename T> cudaError_t launch_pass_d_3d(const PassArgs<T>& a, cudaStream_t s) {
  RVE_DISPATCH_N3(a.n[1], launch_yb_3d_n, a, s)
}
template <typename T> cudaError_t launch_pass_e_3d(const PassArgs<T>& a, cudaStream_t s) {
  RVE_DISPATCH_N3(a.n[0], launch_e_3d_n, a, s)
}

}  // namespace rve

// First pass of the finite elements: material, nodal forces f = B^T sigma in
// real space, and the forward x FFT of the D nodal components.
//
// A block owns TY voxel rows of one z plane over the whole of x and marches
// along y.  A thread owns one column x (3D, FP32: two): per voxel it forms the element
// stresses and the forces of the voxel's 2^D corners (the row below the tile,
// which also acts on the tile's first node row, is computed again: one row in
// TY more).  The corners with dx = 1 go to the next column by a warp shuffle,
// the ones with dy = 1 stay in registers for the next row, so the march has no
// barrier: every warp runs ahead on its own and the loads of the next step are
// in flight while the current one is computed.  At a warp's edge the dx = 1
// corners wait in `edge` and are added after the march.
// 3D: the dz = 0 and dz = 1 corners of the voxel plane z are sums of their own,
// F0 (node plane z) and F1 (node plane z + 1), so no plane is computed twice:
// F0 + i F1 of a node row is one complex row, transformed in place, split by
// the two-for-one rule and stored as components j (F0) and 3 + j (F1, at plane
// z + 1) of the spectrum; pass B adds them when it loads.  2D: f_0 + i f_1.
// Only D (2 D in 3D) components are transformed and stored instead of the m
// stress components.
//
// Source of the corner forces (SRC):
//   S_STRAIN  CG on strain fields: x += alpha_prev p_old, p = r + beta p_old,
//             sigma = C p, <p, sigma> -> alpha (A_CG); or sigma = in (A_BARE).
//             p_old and p_new are different arrays: the row below the tile is
//             read by two blocks.
//             Bound by the 5 m N values per iteration (256 x 256 x 64 in FP32:
//             622 us, 4.9 TB/s of r, p_old, x in and p, x out; a probe that
//             marches the same rows without the arithmetic reaches 5.6: each
//             1 KB row of 36 components opens DRAM pages of its own).
//   S_NODAL   CG on nodal fields: pi = rho + beta pi_old, xi += alpha_prev
//             pi_old, sigma = C B pi, <B pi, sigma> -> alpha.  Bound by issue:
//             about 300 arithmetic instructions per voxel.
//   S_EDGE    rve_apply_operator and its 2D entry point without a handle, whose
//             result leaves the library as it is: sigma = C in (A_FIELD), sigma =
//             in (A_BARE).  The factors of B^H are taken apart, f_j = sum_a
//             d_a^H s_aj, with s_aj the sum of the stresses of the elements at
//             the edge of axis a that starts at the node; the D^2 sums s_aj are
//             transformed, and pass C applies conj(d_a) per wavevector.  In f
//             itself the differences along the short side of a voxel, 1/h_a
//             times larger, leave their rounding error to the wavevectors of
//             the long side (FP32, white noise on the unit cell, 2-norm of the
//             error with f and with s: 1024 x 16 1.1e-6, 2.5e-7; 256 x 16
//             5.3e-7, 2.1e-7; 64 x 64 2.6e-7, 2.1e-7; 16 x 16 x 256 5.2e-7,
//             2.3e-7).  It costs the transforms and the traffic of 9 components
//             instead of 3 (2D: 4 instead of 2): us with f and with s, FP32,
//             256 x 256 x 64: this pass 188, 267, pass B 54, 78, C 97, 108, the
//             call 748, 871; 128^3 486, 551; 1024^2 88, 90.
//             3D: s_x and s_y again in two parts (planes z and z + 1), s_z in
//             one: 15 real rows, 8 complex transforms, components 3 a + j and
//             (second parts) 9 + 3 a + j.
//   S_GRAD    finite strain (2D): the divergence of the stress field in, 4
//             components P_ia per triangle.
#pragma once
#include "pass3d.cuh"

namespace rve {

enum { S_STRAIN = 0, S_NODAL = 1, S_GRAD = 2, S_EDGE = 3 };

// Value of the previous (next) column of the same row; at the row's start (end)
// inside a warp the row wraps, at a warp's first (last) lane of a longer row
// the result is not valid.
template <int NX, typename T> __device__ __forceinline__ T from_prev(T v) {
  if constexpr (NX >= 32) return __shfl_up_sync(0xffffffffu, v, 1);
  else return __shfl_sync(0xffffffffu, v, (threadIdx.x & 31 & ~(NX - 1)) | ((threadIdx.x + NX - 1) & (NX - 1)));
}
template <int NX, typename T> __device__ __forceinline__ T from_next(T v) {
  if constexpr (NX >= 32) return __shfl_down_sync(0xffffffffu, v, 1);
  else return __shfl_sync(0xffffffffu, v, (threadIdx.x & 31 & ~(NX - 1)) | ((threadIdx.x + 1) & (NX - 1)));
}

// ---------------------------------------------------------------- 3D
// Corner forces of tetrahedron t (added to f) from its scaled stress rows.
template <typename T>
__device__ __forceinline__ void tet_forces(int t, const T S[3][3], const T* ih, T f[8][3]) {
  const int pa = kuhn_perm(t, 0), pb = kuhn_perm(t, 1), pc = kuhn_perm(t, 2);
  const int v1 = 1 << pa, v2 = v1 | (1 << pb);
#pragma unroll
  for (int j = 0; j < 3; ++j) {
    const T Pa = ih[pa] * S[pa][j], Pb = ih[pb] * S[pb][j], Pc = ih[pc] * S[pc][j];
    f[0][j] -= Pa;
    f[v1][j] += Pa - Pb;
    f[v2][j] += Pb - Pc;
    f[7][j] += Pc;
  }
}

// Edges of a voxel: the k-th one of axis a starts at the k-th corner without
// bit a (corner dx + 2 dy + 4 dz).
__host__ __device__ constexpr int edge_of(int a, int c) { return a == 0 ? c >> 1 : a == 1 ? (c & 1) + 2 * (c >> 2) : c & 3; }

// Stresses of tetrahedron t, added to the sums g[axis][edge][j] of its three edges.
template <typename T> __device__ __forceinline__ void tet_edges(int t, const T S[3][3], T g[3][4][3]) {
  int at = 0;
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    const int a = kuhn_perm(t, i);
#pragma unroll
    for (int j = 0; j < 3; ++j) g[a][edge_of(a, at)][j] += S[a][j];
    at |= 1 << a;
  }
}

// Corner forces of the six tetrahedra of a voxel from its corner displacements
// and the voxel's share of <B u, C B u>.  Tetrahedra that share an edge share
// its difference (12 edges instead of 18) and its force is summed over them
// before it is scaled and given to the two corners.
template <typename T>
__device__ __forceinline__ T voxel_forces_3d(const T uc[8][3], T e, T lam, T mu2, const T* ih, T f[8][3]) {
  T d[3][4][3];   // d[a][k][j]: difference of u_j along the edge of axis a at the k-th corner without bit a
  auto corner = [](int a, int k) { return a == 0 ? 2 * k : a == 1 ? (k & 1) + 4 * (k >> 1) : k; };
#pragma unroll
  for (int a = 0; a < 3; ++a)
#pragma unroll
    for (int k = 0; k < 4; ++k)
#pragma unroll
      for (int j = 0; j < 3; ++j) d[a][k][j] = (uc[corner(a, k) | (1 << a)][j] - uc[corner(a, k)][j]) * ih[a];
  T S[3][4][3];   // stress sums of the edges
  // the first edge (k = 0) of axis a belongs to tetrahedra 2 a and 2 a + 1, the
  // last (k = 3) to the pair that ends along a; the others to one
  auto put = [](bool more, T* dst, T v0, T v1, T v2) {
    if (more) { dst[0] += v0; dst[1] += v1; dst[2] += v2; }
    else { dst[0] = v0; dst[1] = v1; dst[2] = v2; }
  };
  const T le = e * lam, me = e * mu2, mh = (T)0.5 * me;
  T pq = 0;
#pragma unroll
  for (int t = 0; t < 6; ++t) {
    const int ax[3] = {kuhn_perm(t, 0), kuhn_perm(t, 1), kuhn_perm(t, 2)};
    int ke[3];   // edge index of the tetrahedron's edge along each axis
    int at = 0;
#pragma unroll
    for (int i = 0; i < 3; ++i) { ke[ax[i]] = edge_of(ax[i], at); at |= 1 << ax[i]; }
    const T exx = d[0][ke[0]][0], eyy = d[1][ke[1]][1], ezz = d[2][ke[2]][2];
    const T yz = d[1][ke[1]][2] + d[2][ke[2]][1], xz = d[0][ke[0]][2] + d[2][ke[2]][0];
    const T xy = d[0][ke[0]][1] + d[1][ke[1]][0];
    const T tr = le * (exx + eyy + ezz);
    const T sxx = tr + me * exx, syy = tr + me * eyy, szz = tr + me * ezz;
    const T syz = mh * yz, sxz = mh * xz, sxy = mh * xy;
    pq += exx * sxx + eyy * syy + ezz * szz + yz * syz + xz * sxz + xy * sxy;
    auto more = [&](int a) { return (ke[a] == 0 && t == 2 * a + 1) || (ke[a] == 3 && (t == 2 || t >= 4)); };
    put(more(0), S[0][ke[0]], sxx, sxy, sxz);
    put(more(1), S[1][ke[1]], sxy, syy, syz);
    put(more(2), S[2][ke[2]], sxz, syz, szz);
  }
#pragma unroll
  for (int c = 0; c < 8; ++c)
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      T v = ih[0] * S[0][edge_of(0, c & ~1)][j];
      if (!(c & 1)) v = -v;
#pragma unroll
      for (int a = 1; a < 3; ++a) {
        const T p = S[a][edge_of(a, c & ~(1 << a))][j];
        v = (c >> a) & 1 ? v + ih[a] * p : v - ih[a] * p;
      }
      f[c][j] = v;
    }
  return pq;
}

// Row stride of the transform buffer: 16 / TY (mod 16) complex FP32 values (8 /
// TY mod 8 in FP64), so that the rows that consecutive lanes store, TY at each
// of 16 / TY columns, fall on different banks.
template <typename T, int NX, int TY> __host__ __device__ constexpr int force_ld() {
  constexpr int M = sizeof(T) == 4 ? 16 : 8, want = TY >= M ? 1 : M / TY;
  return FftSplit<NX>::LD + (want - FftSplit<NX>::LD % M + M) % M;
}
// Stages of the ring of the strain and edge sources, and their values a thread each.
template <typename T, int NX, int TY> __host__ __device__ constexpr int force_stages() {
  return NX < 64 && TY == 4 ? 6 : sizeof(T) == 4 ? 3 : 2;
}
template <int SRC> __host__ __device__ constexpr int force_slots() { return SRC == S_STRAIN ? 18 : SRC == S_EDGE ? 6 : 0; }
template <int SRC> __host__ __device__ constexpr int force_rows() { return SRC == S_EDGE ? 8 : 3; }   // complex rows per y
template <typename T, int NX, int TY, int NT, int VL, int SRC> constexpr size_t force_3d_smem() {
  return sizeof(T) * force_stages<T, NX, TY>() * force_slots<SRC>() * NT * VL +
         sizeof(cplx<T>) * force_rows<SRC>() * TY * force_ld<T, NX, TY>() +
         sizeof(T) * 12 * (NX / VL > 32 ? (TY + NT * VL / NX) * (NX / VL / 32) : 0);
}

// grid (n_y/TY, n_z, L).  A thread owns VL neighbouring columns, TPR threads a
// row; NT / TPR rows are marched side by side.
template <typename T, int NX, int TY, int NT, int MB, int VL, int SRC>
__global__ void __launch_bounds__(NT, MB) force_3d(PassArgs<T> a) {
  using C = cplx<T>;
  constexpr int KX = NX / 2 + 1;
  constexpr int LD = force_ld<T, NX, TY>();
  constexpr int TPR = NX / VL;                   // threads per row
  constexpr int LN = NT / TPR, TYL = TY / LN;    // row lanes, rows per lane
  constexpr int NW = TPR > 32 ? TPR / 32 : 1;    // warps per row
  static_assert(NT % TPR == 0 && TY % LN == 0, "threads cover whole rows");
  extern __shared__ __align__(16) unsigned char smem_raw[];
  constexpr bool EDGES = SRC == S_EDGE;
  constexpr int CR = force_rows<SRC>(), SL = force_slots<SRC>();
  C* buf = reinterpret_cast<C*>(smem_raw);                        // [CR][TY][LD]
  T* edge = reinterpret_cast<T*>(buf + CR * TY * LD);             // [LN][TYL + 1][NW][12], TPR > 32
  T* ring = edge + (TPR > 32 ? 12 * (TY + LN) * NW : 0);          // [stages][SL][NT] x VL
  __shared__ double red[NT / 32];
  __shared__ T cols[NT];
  __shared__ int flag;
  const int l = blockIdx.z, z = blockIdx.y, y0 = blockIdx.x * TY;
  const int ny = a.n[1], nz = a.n[2];
  CgState* cg = a.cg + l;
  pdl_begin();
  if (!cg->active) return;
  if (a.cgphase && cg->status != ST_RUN) return;
  const int64_t N = a.N;
  const int tx = threadIdx.x % TPR, ln = threadIdx.x / TPR, x = tx * VL;
  const int lane = threadIdx.x & 31;
  const bool cgm = !EDGES && a.amode == A_CG;
  const bool use_old = cgm && cg->it > 0;
  const T beta = use_old ? cg_beta<T>(cg) : (T)0, alpha_prev = use_old ? cg_alpha<T>(cg) : (T)0;
  const T ih[3] = {a.ih[0], a.ih[1], a.ih[2]};
  const T* Ep = a.E + (int64_t)(l / a.lcs) * N + (int64_t)z * ny * NX + x;
  const int first = ln * TYL - 1, end = (ln + 1) * TYL;
  Acc<T> acc;
  // dy = 1 corners of the row below: [column][dz][j]; edge sums: s_x [dz][j], s_z [2][j]
  constexpr int CY = EDGES ? 3 : 2;
  T carry[VL][CY][3];
#pragma unroll
  for (int k = 0; k < VL; ++k)
#pragma unroll
    for (int j = 0; j < 3 * CY; ++j) carry[k][j / 3][j % 3] = 0;
  auto load_e = [&](int yy, T* e) { vloadn<T, VL>(e, Ep + (int64_t)((y0 + yy) & (ny - 1)) * NX); };

  // corners with dx = 1 of the last column (f: [8][3] corner forces; edge sums
  // [3][4][3]: s_y of dz = 0 and 1, s_z of dy = 0 and 1) -> first column of the
  // next thread
  auto right_of = [&](const T* f, int i, int k, int j) -> T {
    return EDGES ? f[(i + 1) * 12 + (1 + 2 * k) * 3 + j] : f[(1 + 2 * i + 4 * k) * 3 + j];
  };
  auto pass_on = [&](int yy, const T* f, T pv[2][2][3]) {
#pragma unroll
    for (int dy = 0; dy < 2; ++dy)
#pragma unroll
      for (int dz = 0; dz < 2; ++dz)
#pragma unroll
        for (int j = 0; j < 3; ++j) {
          const T u = right_of(f, dy, dz, j);
          T q = from_prev<TPR>(u);
          if constexpr (TPR > 32) {
            if (lane == 31) edge[((ln * (TYL + 1) + yy - first) * NW + tx / 32) * 12 + dy * 6 + dz * 3 + j] = u;
            if (lane == 0) q = 0;
          } else if constexpr (TPR == 32) {
            const T w = __shfl_sync(0xffffffffu, u, 31);
            if (lane == 0) q = w;
          }
          pv[dy][dz][j] = q;
        }
  };
  // column k of row yy: corners dx = 0 of its voxel (f) and dx = 1 of the voxel before (pv)
  auto put_column = [&](int yy, int k, const T* f, const T pv[2][2][3]) {
    const bool own = yy > first;
    if constexpr (EDGES) {
      auto g = [&](int ax, int e, int j) -> T { return f[ax * 12 + e * 3 + j]; };
      T sz[3];
#pragma unroll
      for (int j = 0; j < 3; ++j) {
        const C sx = mkc<T>(g(0, 0, j) + carry[k][0][j], g(0, 2, j) + carry[k][1][j]);   // x edges dy + 2 dz
        const C sy = mkc<T>(g(1, 0, j) + pv[0][0][j], g(1, 2, j) + pv[0][1][j]);         // y edges dx + 2 dz
        sz[j] = g(2, 0, j) + pv[1][0][j] + carry[k][2][j];                               // z edges dx + 2 dy
        carry[k][0][j] = g(0, 1, j);
        carry[k][1][j] = g(0, 3, j);
        carry[k][2][j] = g(2, 2, j) + pv[1][1][j];
        if (own) {
          buf[(j * TY + yy) * LD + x + k] = sx;
          buf[((3 + j) * TY + yy) * LD + x + k] = sy;
        }
      }
      if (own) {
        buf[(6 * TY + yy) * LD + x + k] = mkc<T>(sz[0], sz[1]);
        buf[(7 * TY + yy) * LD + x + k] = mkc<T>(sz[2], (T)0);
      }
    } else {
      T v[2][3];
#pragma unroll
      for (int dz = 0; dz < 2; ++dz)
#pragma unroll
        for (int j = 0; j < 3; ++j) {
          v[dz][j] = f[12 * dz + j] + pv[0][dz][j] + carry[k][dz][j];
          carry[k][dz][j] = f[6 + 12 * dz + j] + pv[1][dz][j];
        }
      if (own) {
#pragma unroll
        for (int j = 0; j < 3; ++j) buf[(j * TY + yy) * LD + x + k] = mkc<T>(v[0][j], v[1][j]);
      }
    }
  };
  auto right = [&](const T* f, T pv[2][2][3]) {   // within the thread
#pragma unroll
    for (int dy = 0; dy < 2; ++dy)
#pragma unroll
      for (int dz = 0; dz < 2; ++dz)
#pragma unroll
        for (int j = 0; j < 3; ++j) pv[dy][dz][j] = right_of(f, dy, dz, j);
  };

  if constexpr (SRC == S_STRAIN || SRC == S_EDGE) {
    // A step is one tetrahedron of one row: 6 values each of r, p_old and x
    // (edge source: of the field in).
    // Every thread copies its own values of the next ST - 1 steps into its own
    // slots of the ring (cp.async: no registers are held, and since no thread
    // reads another's slot there is no barrier).
    constexpr int ST = force_stages<T, NX, TY>();
    static_assert(6 % ST == 0, "step t of every row uses slot t % ST");
    const int64_t base = (int64_t)l * a.m * N + (int64_t)z * ny * NX;
    const T* rp = (cgm ? a.r : a.in) + base;
    const T* po = a.pold + base;
    T* pn = a.pnew + base;
    T* xp = a.x + base;
    const bool mat = a.amode != A_BARE;
    auto off = [&](int yy) -> unsigned { return (unsigned)(((y0 + yy) & (ny - 1)) * NX + x); };
    auto slot = [&](int t, int s) -> T* { return ring + (((t % ST) * SL + s) * NT + threadIdx.x) * VL; };
    auto issue = [&](int yy, int t) {   // step (yy, t) into slot t % ST
      if (yy < end) {
        const unsigned o = off(yy);
        constexpr int B = VL * (int)sizeof(T);
#pragma unroll
        for (int s = 0; s < 6; ++s) copy_async<B>(slot(t, s), rp + (6 * t + s) * N + o);
        if (!EDGES && use_old) {
#pragma unroll
          for (int s = 0; s < 6; ++s) copy_async<B>(slot(t, 6 + s), po + (6 * t + s) * N + o);
          if (yy > first) {
#pragma unroll
            for (int s = 0; s < 6; ++s) copy_async<B>(slot(t, 12 + s), xp + (6 * t + s) * N + o);
          }
        }
      }
      copy_async_commit();
    };
    const T r2 = (T)kInvSqrt2;
#pragma unroll
    for (int t = 0; t < ST - 1; ++t) issue(first, t);
    T e[VL], en[VL];
#pragma unroll
    for (int k = 0; k < VL; ++k) e[k] = en[k] = 1;
    if (mat) load_e(first, e);
    for (int yy = first; yy < end; ++yy) {
      const bool own = yy > first;
      const unsigned o = off(yy);
      if (mat && yy + 1 < end) load_e(yy + 1, en);
      constexpr int NF = EDGES ? 36 : 24;   // edge sums [3][4][3] or corner forces [8][3]
      T f[VL][NF];
#pragma unroll
      for (int k = 0; k < VL; ++k)
#pragma unroll
        for (int c = 0; c < NF; ++c) f[k][c] = 0;
      T pq = 0;
#pragma unroll
      for (int t = 0; t < 6; ++t) {
        issue(t + ST - 1 < 6 ? yy : yy + 1, (t + ST - 1) % 6);
        copy_async_wait<ST - 1>();
        T p[6][VL];
#pragma unroll
        for (int s = 0; s < 6; ++s) vloadn<T, VL>(p[s], slot(t, s));
        if (!EDGES && use_old) {
#pragma unroll
          for (int s = 0; s < 6; ++s) {
            T v[VL];
            vloadn<T, VL>(v, slot(t, 6 + s));
#pragma unroll
            for (int k = 0; k < VL; ++k) p[s][k] += beta * v[k];
            if (own) {
              T xv[VL];
              vloadn<T, VL>(xv, slot(t, 12 + s));
#pragma unroll
              for (int k = 0; k < VL; ++k) xv[k] += alpha_prev * v[k];
              vstoren<T, VL>(xp + (6 * t + s) * N + o, xv);
            }
          }
        }
        if (cgm && own) {
#pragma unroll
          for (int s = 0; s < 6; ++s) vstoren<T, VL>(pn + (6 * t + s) * N + o, p[s]);
        }
#pragma unroll
        for (int k = 0; k < VL; ++k) {
          T sg[6];
          if (mat) {
            const T tr = e[k] * (a.lam * (p[0][k] + p[1][k] + p[2][k])), me = e[k] * a.mu2;
#pragma unroll
            for (int s = 0; s < 6; ++s) sg[s] = s < 3 ? tr + me * p[s][k] : me * p[s][k];
#pragma unroll
            for (int s = 0; s < 6; ++s) pq += EDGES ? (T)0 : p[s][k] * sg[s];
          } else {
#pragma unroll
            for (int s = 0; s < 6; ++s) sg[s] = p[s][k];
          }
          T S[3][3];
          S[0][0] = sg[0]; S[1][1] = sg[1]; S[2][2] = sg[2];
          S[1][2] = S[2][1] = r2 * sg[3]; S[0][2] = S[2][0] = r2 * sg[4]; S[0][1] = S[1][0] = r2 * sg[5];
          if constexpr (EDGES) tet_edges<T>(t, S, reinterpret_cast<T(*)[4][3]>(f[k]));
          else tet_forces<T>(t, S, ih, reinterpret_cast<T(*)[3]>(f[k]));
        }
      }
      if (!EDGES && own) acc.add(pq);
      T pv[2][2][3];
      pass_on(yy, f[VL - 1], pv);
#pragma unroll
      for (int k = 0; k < VL; ++k) {
        put_column(yy, k, f[k], pv);
        right(f[k], pv);
      }
#pragma unroll
      for (int k = 0; k < VL; ++k) e[k] = en[k];
    }
    copy_async_wait<0>();
  } else {
    const int64_t lb = (int64_t)l * 3 * N;
    const int64_t plane = (int64_t)ny * NX;
    const int64_t zo[2] = {lb + (int64_t)z * plane, lb + (int64_t)((z + 1) & (nz - 1)) * plane};
    const T* __restrict__ rho = a.rho;
    const T* __restrict__ po = a.pold;
    T* __restrict__ pn = a.pnew;
    T* __restrict__ xi = a.xi;
    const bool last = TPR > 32 && lane == 31;   // the next column belongs to another warp
    // values of node row yy in flight: planes z and z + 1, own columns and (last
    // lane) the next one; p_old counts as 0 in the first iteration
    T rv[2][3][VL], pv[2][3][VL], xv[3][VL], re[2][3], pe[2][3];
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      re[0][j] = re[1][j] = pe[0][j] = pe[1][j] = 0;
#pragma unroll
      for (int k = 0; k < VL; ++k) pv[0][j][k] = pv[1][j][k] = xv[j][k] = 0;
    }
    auto fetch = [&](int yy) {
      const unsigned row = (unsigned)(((y0 + yy) & (ny - 1)) * NX), o = row + x;
#pragma unroll
      for (int dz = 0; dz < 2; ++dz)
#pragma unroll
        for (int j = 0; j < 3; ++j) {
          vloadn<T, VL>(rv[dz][j], rho + zo[dz] + j * N + o);
          if (use_old) vloadn<T, VL>(pv[dz][j], po + zo[dz] + j * N + o);
        }
      if (last) {
        const unsigned on = row + ((x + VL) & (NX - 1));
#pragma unroll
        for (int dz = 0; dz < 2; ++dz)
#pragma unroll
          for (int j = 0; j < 3; ++j) {
            re[dz][j] = (rho + zo[dz] + j * N)[on];
            if (use_old) pe[dz][j] = (po + zo[dz] + j * N)[on];
          }
      }
      if (use_old && yy > first && yy < end) {
#pragma unroll
        for (int j = 0; j < 3; ++j) vloadn<T, VL>(xv[j], xi + zo[0] + j * N + o);
      }
    };
    // pi of node row yy at columns x .. x + VL: u[dz][column][j]
    auto commit = [&](int yy, T u[2][VL + 1][3]) {
#pragma unroll
      for (int dz = 0; dz < 2; ++dz)
#pragma unroll
        for (int j = 0; j < 3; ++j) {
#pragma unroll
          for (int k = 0; k < VL; ++k) u[dz][k][j] = rv[dz][j][k] + beta * pv[dz][j][k];
          T q = from_next<TPR>(u[dz][0][j]);
          if constexpr (TPR > 32) {
            if (last) q = re[dz][j] + beta * pe[dz][j];
          } else if constexpr (TPR == 32) {
            const T w = __shfl_sync(0xffffffffu, u[dz][0][j], 0);
            if (lane == 31) q = w;
          }
          u[dz][VL][j] = q;
        }
      if (yy > first && yy < end) {
        const unsigned o = (unsigned)(((y0 + yy) & (ny - 1)) * NX + x);
#pragma unroll
        for (int j = 0; j < 3; ++j) {
          T s[VL];
#pragma unroll
          for (int k = 0; k < VL; ++k) s[k] = u[0][k][j];
          vstoren<T, VL>(pn + zo[0] + j * N + o, s);
          if (use_old) {
#pragma unroll
            for (int k = 0; k < VL; ++k) s[k] = xv[j][k] + alpha_prev * pv[0][j][k];
            vstoren<T, VL>(xi + zo[0] + j * N + o, s);
          }
        }
      }
    };
    T lo[2][VL + 1][3], hi[2][VL + 1][3];
    fetch(first);
    commit(first, lo);
    fetch(first + 1);
    T e[VL], en[VL];
    load_e(first, e);
#pragma unroll
    for (int k = 0; k < VL; ++k) en[k] = 0;
    for (int yy = first; yy < end; ++yy) {
      commit(yy + 1, hi);
      if (yy + 1 < end) {
        fetch(yy + 2);
        load_e(yy + 1, en);
      }
      const bool own = yy > first;
      T pq = 0, keep[2][2][3], f[8][3], pv1[2][2][3];
      // from the last column back, so that one column's forces are live at a time:
      // its dx = 0 corners wait in keep for the dx = 1 corners of the column before
#pragma unroll
      for (int k = VL - 1; k >= 0; --k) {
        T uc[8][3];
#pragma unroll
        for (int c = 0; c < 8; ++c)
#pragma unroll
          for (int j = 0; j < 3; ++j) uc[c][j] = ((c >> 1) & 1 ? hi : lo)[c >> 2][k + (c & 1)][j];
        pq += voxel_forces_3d<T>(uc, e[k], a.lam, a.mu2, ih, f);
        if (k == VL - 1) pass_on(yy, f[0], pv1);
        if (k < VL - 1) {   // finish column k + 1
          T g[8][3], pr[2][2][3];
          right(f[0], pr);
#pragma unroll
          for (int dy = 0; dy < 2; ++dy)
#pragma unroll
            for (int dz = 0; dz < 2; ++dz)
#pragma unroll
              for (int j = 0; j < 3; ++j) g[2 * dy + 4 * dz][j] = keep[dy][dz][j];
          put_column(yy, k + 1, g[0], pr);
        }
#pragma unroll
        for (int dy = 0; dy < 2; ++dy)
#pragma unroll
          for (int dz = 0; dz < 2; ++dz)
#pragma unroll
            for (int j = 0; j < 3; ++j) keep[dy][dz][j] = f[2 * dy + 4 * dz][j];
      }
      put_column(yy, 0, f[0], pv1);
      if (own) acc.add(pq);
#pragma unroll
      for (int k = 0; k < VL; ++k) e[k] = en[k];
#pragma unroll
      for (int dz = 0; dz < 2; ++dz)
#pragma unroll
        for (int c = 0; c <= VL; ++c)
#pragma unroll
          for (int j = 0; j < 3; ++j) lo[dz][c][j] = hi[dz][c][j];
    }
  }

  __syncthreads();
  if constexpr (TPR > 32) {
    for (int i = threadIdx.x; i < (EDGES ? 5 : 3) * TY * NW; i += NT) {
      const int w = i % NW, yy = (i / NW) % TY, j = i / (NW * TY);
      const int q = yy / TYL, lr = yy % TYL + 1;   // the lane's rows: 0 is the row below its first
      const int wp = (w + NW - 1) % NW;
      const T* r0 = edge + ((q * (TYL + 1) + lr) * NW + wp) * 12;        // dy = 0 of row yy
      const T* r1 = edge + ((q * (TYL + 1) + lr - 1) * NW + wp) * 12;    // dy = 1 of row yy - 1
      if constexpr (EDGES) {   // j < 3: s_y; 3, 4: the two rows of s_z
        C* p = buf + ((3 + j) * TY + yy) * LD + 32 * VL * w;
        if (j < 3) *p = mkc<T>(p->x + r0[j], p->y + r0[3 + j]);
        else if (j == 3) *p = mkc<T>(p->x + r0[6] + r1[9], p->y + r0[7] + r1[10]);
        else p->x += r0[8] + r1[11];
      } else {
        C* p = buf + (j * TY + yy) * LD + 32 * VL * w;
        *p = mkc<T>(p->x + r0[j] + r1[6 + j], p->y + r0[3 + j] + r1[9 + j]);
      }
    }
    __syncthreads();
  }
  smem_fft<T, NX, CR * TY, LD, NT, -1>(buf, a.tw[0]);
  if constexpr (EDGES) {
    const int64_t cs = (int64_t)KX * nz * ny;
    C* p0 = a.spec + (int64_t)l * a.m * cs + (int64_t)z * ny + y0;
    C* p1 = a.spec + (int64_t)l * a.m * cs + (int64_t)((z + 1) & (nz - 1)) * ny + y0;
    for (int i = threadIdx.x; i < 8 * KX * TY; i += NT) {
      const int yy = i % TY, k = (i / TY) % KX, j = i / (TY * KX);
      const C* row = buf + (j * TY + yy) * LD;
      const C A = row[k], B = cconj(row[(NX - k) & (NX - 1)]);
      const C d = csub(A, B);
      const int64_t o = (int64_t)k * nz * ny + yy;
      p0[(j == 7 ? 8 : j) * cs + o] = cscale(cadd(A, B), (T)0.5);
      const C im = mkc<T>((T)0.5 * d.y, (T)-0.5 * d.x);
      if (j < 6) p1[(9 + j) * cs + o] = im;
      else if (j == 6) p0[7 * cs + o] = im;
    }
  } else {
    C* s0 = a.spec + ((int64_t)l * a.m * KX * nz + z) * ny + y0;
    C* s1 = a.spec + ((((int64_t)l * a.m + 3) * KX) * nz + ((z + 1) & (nz - 1))) * ny + y0;
    for (int i = threadIdx.x; i < 3 * KX * TY; i += NT) {
      const int yy = i % TY, k = (i / TY) % KX, j = i / (TY * KX);
      const C* row = buf + (j * TY + yy) * LD;
      const C A = row[k], B = cconj(row[(NX - k) & (NX - 1)]);
      const C d = csub(A, B);
      const int64_t o = ((int64_t)j * KX + k) * nz * ny + yy;
      s0[o] = cscale(cadd(A, B), (T)0.5);
      s1[o] = mkc<T>((T)0.5 * d.y, (T)-0.5 * d.x);
    }
  }
  if (cgm) {
    const double s = block_sum_acc<NT>(acc, cols);
    const int nblk = gridDim.x * gridDim.y, blk = blockIdx.x + gridDim.x * blockIdx.y;
    double* part = a.part + (int64_t)l * a.part_stride;
    if (publish_partial(s, part, &cg->cnt_a, blk, nblk, &flag)) {
      const double pq = sum_partials<NT>(part, nblk, red);
      if (threadIdx.x == 0) finish_alpha(cg, pq);
    }
  }
}

// ---------------------------------------------------------------- 2D
// Corner forces f[c][j], c = dx + 2 dy, of the two triangles of a pixel from
// their stresses S[q] = (xx, yy, xy).
template <typename T>
__device__ __forceinline__ void pixel_forces(const T S[2][3], T ihx, T ihy, T f[4][2]) {
  // element 0 = nodes {00, 10, 01}: grad N_00 = (-ihx, -ihy), N_10 = (ihx, 0), N_01 = (0, ihy)
  // element 1 = nodes {11, 01, 10}: grad N_11 = (ihx, ihy), N_01 = (-ihx, 0), N_10 = (0, -ihy)
  f[0][0] = -ihx * S[0][0] - ihy * S[0][2];
  f[0][1] = -ihx * S[0][2] - ihy * S[0][1];
  f[1][0] = ihx * S[0][0] - ihy * S[1][2];
  f[1][1] = ihx * S[0][2] - ihy * S[1][1];
  f[2][0] = ihy * S[0][2] - ihx * S[1][0];
  f[2][1] = ihy * S[0][1] - ihx * S[1][2];
  f[3][0] = ihx * S[1][0] + ihy * S[1][2];
  f[3][1] = ihx * S[1][2] + ihy * S[1][1];
}

// The same pixel's stresses at the edges they act on, f[c][2 a + j] = s_aj of
// corner c: element 0 has its x and y edges at the pixel's own node, element 1
// the x edge at corner dy = 1 and the y edge at corner dx = 1.  S[q][a][j].
template <typename T> __device__ __forceinline__ void pixel_edges(const T S[2][2][2], T f[4][4]) {
#pragma unroll
  for (int j = 0; j < 2; ++j) {
    f[0][j] = S[0][0][j];
    f[0][2 + j] = S[0][1][j];
    f[1][j] = 0;
    f[1][2 + j] = S[1][1][j];
    f[2][j] = S[1][0][j];
    f[2][2 + j] = f[3][j] = f[3][2 + j] = 0;
  }
}

// Real rows of a node row: the forces f_j or the edge sums s_aj.
template <int SRC> __host__ __device__ constexpr int force_comps2() { return SRC == S_EDGE ? 4 : 2; }
template <typename T, int NX, int TY, int LN, int NC> constexpr size_t force_2d_smem() {
  return sizeof(cplx<T>) * (NC / 2) * TY * force_ld<T, NX, TY>() +
         sizeof(T) * 2 * NC * (NX > 32 ? (TY + LN) * (NX / 32) : 0);
}

// The same for a field of first Piola-Kirchhoff stresses P[q][i][a] (finite
// strain; not symmetric).
template <typename T>
__device__ __forceinline__ void pixel_divergence(const T P[8], T ihx, T ihy, T f[4][2]) {
#pragma unroll
  for (int i = 0; i < 2; ++i) {
    const T x0 = ihx * P[2 * i], y0 = ihy * P[2 * i + 1], x1 = ihx * P[4 + 2 * i], y1 = ihy * P[5 + 2 * i];
    f[0][i] = -x0 - y0;
    f[1][i] = x0 - y1;
    f[2][i] = y0 - x1;
    f[3][i] = x1 + y1;
  }
}

// grid (n_y/TY, L).  NT < NX: a thread marches NX / NT columns one after the
// other; NT > NX: NT / NX rows side by side.
template <typename T, int NX, int TY, int NT, int MB, int SRC>
__global__ void __launch_bounds__(NT, MB) force_2d(PassArgs<T> a) {
  using C = cplx<T>;
  constexpr int KX = NX / 2 + 1;
  constexpr int LD = force_ld<T, NX, TY>();
  constexpr int CPT = NX > NT ? NX / NT : 1;
  constexpr int LN = NT > NX ? NT / NX : 1, TYL = TY / LN;
  constexpr int NW = NX > 32 ? NX / 32 : 1;
  static_assert((NT % NX == 0 || NX % NT == 0) && TY % LN == 0, "threads cover whole rows");
  extern __shared__ __align__(16) unsigned char smem_raw[];
  constexpr int NC = force_comps2<SRC>();
  constexpr bool EDGES = NC == 4;
  C* buf = reinterpret_cast<C*>(smem_raw);             // [NC / 2][TY][LD]: f_0 + i f_1, or s_a0 + i s_a1
  T* edge = reinterpret_cast<T*>(buf + NC / 2 * TY * LD);   // [LN][TYL + 1][NW][2 NC], NX > 32
  __shared__ double red[NT / 32];
  __shared__ T cols[NT];
  __shared__ int flag;
  const int l = blockIdx.y, y0 = blockIdx.x * TY;
  const int ny = a.n[1];
  CgState* cg = a.cg + l;
  pdl_begin();
  if (!cg->active) return;
  if (a.cgphase && cg->status != ST_RUN) return;
  const int64_t N = a.N;
  const int ln = LN > 1 ? threadIdx.x / NX : 0, lane = threadIdx.x & 31;
  const bool cgm = !EDGES && a.amode == A_CG;
  const bool use_old = cgm && cg->it > 0;
  const T beta = cgm ? cg_beta<T>(cg) : (T)0, alpha_prev = cgm ? cg_alpha<T>(cg) : (T)0;
  const T ihx = a.ih[0], ihy = a.ih[1], r2 = (T)kInvSqrt2;
  const int first = ln * TYL - 1, end = (ln + 1) * TYL;
  Acc<T> acc;
#pragma unroll 1
  for (int cx = 0; cx < CPT; ++cx) {
    const int x = LN > 1 ? threadIdx.x % NX : cx * NT + threadIdx.x;
    const T* Ep = a.E + (int64_t)(l / a.lcs) * N + x;
    T carry[NC];
#pragma unroll
    for (int j = 0; j < NC; ++j) carry[j] = 0;
    auto node_row = [&](int yy, const T f[4][NC], bool own) {
      T s[2][NC];   // [dy][j]
#pragma unroll
      for (int dy = 0; dy < 2; ++dy)
#pragma unroll
        for (int j = 0; j < NC; ++j) {
          if (EDGES && (dy == 1 || j < 2)) {   // nothing at dx = 1 (see pixel_edges)
            s[dy][j] = f[2 * dy][j];
            continue;
          }
          const T u = f[1 + 2 * dy][j];
          T p = from_prev<NX>(u);
          if constexpr (NX > 32) {
            if (lane == 31) edge[((ln * (TYL + 1) + yy + 1 - ln * TYL) * NW + x / 32) * 2 * NC + dy * NC + j] = u;
            if (lane == 0) p = 0;
          } else if constexpr (NX == 32) {
            const T w = __shfl_sync(0xffffffffu, u, 31);
            if (lane == 0) p = w;
          }
          s[dy][j] = f[2 * dy][j] + p;
        }
      if (own) {
#pragma unroll
        for (int c = 0; c < NC / 2; ++c)
          buf[(c * TY + yy) * LD + x] = mkc<T>(s[0][2 * c] + carry[2 * c], s[0][2 * c + 1] + carry[2 * c + 1]);
      }
#pragma unroll
      for (int j = 0; j < NC; ++j) carry[j] = s[1][j];
    };
    if constexpr (SRC == S_GRAD) {
      const T* __restrict__ in = a.in + (int64_t)l * a.m * N + x;
      for (int yy = first; yy < end; ++yy) {
        const int64_t o = (int64_t)((y0 + yy) & (ny - 1)) * NX;
        T P[8], f[4][2];
#pragma unroll
        for (int s = 0; s < 8; ++s) P[s] = in[o + s * N];
        pixel_divergence<T>(P, ihx, ihy, f);
        node_row(yy, f, yy >= ln * TYL);
      }
    } else if constexpr (SRC == S_STRAIN || SRC == S_EDGE) {
      const int64_t base = (int64_t)l * a.m * N + x;
      const T* __restrict__ rp = (cgm ? a.r : a.in) + base;
      const T* __restrict__ po = a.pold + base;
      T* __restrict__ pn = a.pnew + base;
      T* xp = a.x + base;
      const bool mat = a.amode != A_BARE;
      T rv[6], pv[6], xv[6], e = 1;
      auto fetch = [&](int yy) {
        const int64_t o = (int64_t)((y0 + yy) & (ny - 1)) * NX;
#pragma unroll
        for (int s = 0; s < 6; ++s) rv[s] = rp[o + s * N];
        if (use_old) {
#pragma unroll
          for (int s = 0; s < 6; ++s) pv[s] = po[o + s * N];
          if (yy >= ln * TYL) {
#pragma unroll
            for (int s = 0; s < 6; ++s) xv[s] = xp[o + s * N];
          }
        }
        if (mat) e = Ep[o];
      };
      fetch(first);
      for (int yy = first; yy < end; ++yy) {
        const bool own = yy >= ln * TYL;
        const int64_t o = (int64_t)((y0 + yy) & (ny - 1)) * NX;
        T p[6], xs[6];
        const T ec = e;
#pragma unroll
        for (int s = 0; s < 6; ++s) {
          p[s] = use_old ? rv[s] + beta * pv[s] : rv[s];
          xs[s] = use_old ? xv[s] + alpha_prev * pv[s] : (T)0;
        }
        if (yy + 1 < end) fetch(yy + 1);
        if (cgm && own) {
#pragma unroll
          for (int s = 0; s < 6; ++s) pn[o + s * N] = p[s];
          if (use_old) {
#pragma unroll
            for (int s = 0; s < 6; ++s) xp[o + s * N] = xs[s];
          }
        }
        T S[2][3], f[4][NC], pq = 0;
#pragma unroll
        for (int q = 0; q < 2; ++q) {
          if (mat) {
            const T tr = ec * (a.lam * (p[3 * q] + p[3 * q + 1])), me = ec * a.mu2;
            S[q][0] = tr + me * p[3 * q];
            S[q][1] = tr + me * p[3 * q + 1];
            S[q][2] = me * p[3 * q + 2];
            pq += p[3 * q] * S[q][0] + p[3 * q + 1] * S[q][1] + p[3 * q + 2] * S[q][2];
            S[q][2] *= r2;
          } else {
            S[q][0] = p[3 * q]; S[q][1] = p[3 * q + 1]; S[q][2] = r2 * p[3 * q + 2];
          }
        }
        if constexpr (EDGES) {
          const T G[2][2][2] = {{{S[0][0], S[0][2]}, {S[0][2], S[0][1]}}, {{S[1][0], S[1][2]}, {S[1][2], S[1][1]}}};
          pixel_edges<T>(G, f);
        } else {
          pixel_forces<T>(S, ihx, ihy, f);
          if (own) acc.add(pq);
        }
        node_row(yy, f, own);
      }
    } else {
      const int64_t lb = (int64_t)l * 2 * N;
      const T* __restrict__ rho = a.rho + lb;
      const T* __restrict__ po = a.pold + lb;
      T* __restrict__ pn = a.pnew + lb;
      T* __restrict__ xi = a.xi + lb;
      const int xn = (x + 1) & (NX - 1);
      const bool last = NX > 32 && lane == 31;
      T rv[2], pv[2], xv[2], re[2], pe[2];
      auto fetch = [&](int yy) {
        const int64_t ro = (int64_t)((y0 + yy) & (ny - 1)) * NX;
#pragma unroll
        for (int j = 0; j < 2; ++j) {
          rv[j] = rho[j * N + ro + x];
          if (use_old) pv[j] = po[j * N + ro + x];
          if (last) {
            re[j] = rho[j * N + ro + xn];
            if (use_old) pe[j] = po[j * N + ro + xn];
          }
          if (use_old && yy >= ln * TYL && yy < end) xv[j] = xi[j * N + ro + x];
        }
      };
      // pi of node row yy at columns x and x + 1: u[dx][j]
      auto commit = [&](int yy, T u[2][2]) {
#pragma unroll
        for (int j = 0; j < 2; ++j) {
          const T p = use_old ? rv[j] + beta * pv[j] : rv[j];
          u[0][j] = p;
          T q = from_next<NX>(p);
          if constexpr (NX > 32) {
            const T w = use_old ? re[j] + beta * pe[j] : re[j];
            if (last) q = w;
          } else if constexpr (NX == 32) {
            const T w = __shfl_sync(0xffffffffu, p, 0);
            if (lane == 31) q = w;
          }
          u[1][j] = q;
        }
        if (yy >= ln * TYL && yy < end) {
          const int64_t o = (int64_t)((y0 + yy) & (ny - 1)) * NX + x;
#pragma unroll
          for (int j = 0; j < 2; ++j) {
            pn[j * N + o] = u[0][j];
            if (use_old) xi[j * N + o] = xv[j] + alpha_prev * pv[j];
          }
        }
      };
      T lo[2][2], hi[2][2];
      fetch(first);
      commit(first, lo);
      fetch(first + 1);
      T e = Ep[(int64_t)((y0 + first) & (ny - 1)) * NX];
      for (int yy = first; yy < end; ++yy) {
        commit(yy + 1, hi);
        T en = 0;
        if (yy + 1 < end) {
          fetch(yy + 2);
          en = Ep[(int64_t)((y0 + yy + 1) & (ny - 1)) * NX];
        }
        T S[2][3], f[4][2], pq = 0;
        const T le = e * a.lam, me = e * a.mu2, mh = (T)0.5 * me;
        // element 0: d/dx = u10 - u00, d/dy = u01 - u00; element 1: u11 - u01, u11 - u10
#pragma unroll
        for (int q = 0; q < 2; ++q) {
          const T* bx = q ? hi[0] : lo[0];
          const T* tx = q ? hi[1] : lo[1];
          const T* by = q ? lo[1] : lo[0];
          const T* ty = q ? hi[1] : hi[0];
          const T exx = (tx[0] - bx[0]) * ihx, eyy = (ty[1] - by[1]) * ihy;
          const T xy = (ty[0] - by[0]) * ihy + (tx[1] - bx[1]) * ihx;
          const T tr = le * (exx + eyy);
          S[q][0] = tr + me * exx;
          S[q][1] = tr + me * eyy;
          S[q][2] = mh * xy;
          pq += exx * S[q][0] + eyy * S[q][1] + xy * S[q][2];
        }
        pixel_forces<T>(S, ihx, ihy, f);
        const bool own = yy >= ln * TYL;
        if (own) acc.add(pq);
        node_row(yy, f, own);
        e = en;
#pragma unroll
        for (int c = 0; c < 2; ++c) { lo[c][0] = hi[c][0]; lo[c][1] = hi[c][1]; }
      }
    }
  }
  __syncthreads();
  if constexpr (NX > 32) {
    for (int i = threadIdx.x; i < TY * NW; i += NT) {
      const int w = i % NW, yy = i / NW, q = yy / TYL, lr = yy % TYL + 1, wp = (w + NW - 1) % NW;
      const T* r0 = edge + ((q * (TYL + 1) + lr) * NW + wp) * 2 * NC;            // dy = 0 of row yy
      const T* r1 = edge + ((q * (TYL + 1) + lr - 1) * NW + wp) * 2 * NC + NC;   // dy = 1 of row yy - 1
      C* p = buf + ((EDGES ? TY : 0) + yy) * LD + 32 * w;                        // edge sums: s_y only
      if constexpr (EDGES) *p = mkc<T>(p->x + r0[2], p->y + r0[3]);
      else *p = mkc<T>(p->x + r0[0] + r1[0], p->y + r0[1] + r1[1]);
    }
    __syncthreads();
  }
  if constexpr (!EDGES && sizeof(T) == 4 && (NX == 512 || NX == 1024) && NT == 2 * FftSplit<NX>::N1 * TY)
    smem_fft_pair<T, NX, TY, LD, NT, -1>(buf, a.tw[0]);
  else
    smem_fft<T, NX, NC / 2 * TY, LD, NT, -1>(buf, a.tw[0]);
  {
    C* s0 = a.spec + (int64_t)l * a.m * KX * ny + y0;
    for (int i = threadIdx.x; i < NC / 2 * KX * TY; i += NT) {
      const int yy = i % TY, k = (i / TY) % KX, c = i / (TY * KX);
      const C* row = buf + (c * TY + yy) * LD;
      const C A = row[k], B = cconj(row[(NX - k) & (NX - 1)]);
      const C d = csub(A, B);
      C* o = s0 + ((int64_t)2 * c * KX + k) * ny + yy;
      o[0] = cscale(cadd(A, B), (T)0.5);
      o[(int64_t)KX * ny] = mkc<T>((T)0.5 * d.y, (T)-0.5 * d.x);
    }
  }
  if (cgm) {
    const double s = block_sum_acc<NT>(acc, cols);
    double* part = a.part + (int64_t)l * a.part_stride;
    if (publish_partial(s, part, &cg->cnt_a, blockIdx.x, gridDim.x, &flag)) {
      const double pq = sum_partials<NT>(part, gridDim.x, red);
      if (threadIdx.x == 0) finish_alpha(cg, pq);
    }
  }
}

// ------------------------------------------------------------ launchers
template <typename T, int NX, int TY, int NT, int VL, int SRC>
cudaError_t launch_force_3d_t(const PassArgs<T>& a, cudaStream_t s) {
  // resident blocks the registers are sized for (shared memory holds two of the
  // strain source's 128-thread blocks)
  constexpr int MB = sizeof(T) == 8 ? 1 : VL == 2 ? (NT <= 64 ? 2 : 1) * (SRC == S_NODAL ? 3 : 2) / (NT <= 128 ? 1 : 2)
                                         : NT <= 64 ? 8 : NT <= 128 ? 4 : NT <= 256 ? 2 : 1;
  constexpr size_t sm = force_3d_smem<T, NX, TY, NT, VL, SRC>();
  static_assert(sm <= 222 * 1024, "shared memory of the tile");
  auto k = force_3d<T, NX, TY, NT, MB, VL, SRC>;
  static DeviceOnce attr;
  attr.run(current_device(), [&] { set_smem_attrs(k, sm); });
  return launch_pass(a.pdl, k, dim3(a.n[1] / TY, a.n[2], a.L), NT, sm, s, a);
}
// Columns per thread: two in FP32 where a row still fills a warp (8-byte
// accesses: half the load and store instructions, which throttled the pass, and
// half the shuffles).  us per iteration, one and two columns: strain source 256 x
// 256 x 64 657, 622, 64^3 (six load cases) 265, 253, 128^3 342, 341; nodal source
// 256 x 256 x 128 319, 248, 64^3 71, 58, 128^3 (two) 187, 164.
template <typename T, int NX> constexpr int force_cols3() { return sizeof(T) == 4 && NX >= 64 ? 2 : 1; }
// Rows per block and threads.  Long rows need the shared memory for fewer of
// them; short ones are marched side by side, with few rows per lane.
template <typename T, int NX> constexpr int force_rows3() { return NX >= 128 ? 8 : 16; }
template <int NX, int VL> constexpr int force_threads3() { return (NX >= 256 ? 256 : NX >= 64 ? 128 : 64) / (NX >= 64 ? VL : 1); }
// Tile variants: 0 default rows, 1 half, 2 double (n_x >= 128: 16 rows, FP32),
// 3 and 4 the rows of 0 and 1 with twice the threads; 6 as 0 (an L2 prefetch of
// the rows two steps ahead, 2 KB of each of the 108 fields, made the pass
// slower: 256 x 256 x 64 657 -> 770 us).
template <typename T, int NX>
cudaError_t launch_force_3d_n(const PassArgs<T>& a, cudaStream_t s) {
  constexpr int TY = force_rows3<T, NX>();
  constexpr int VS = force_cols3<T, NX>();
  constexpr int NT = force_threads3<NX, VS>();
  if (a.force == 2) return launch_force_3d_t<T, NX, TY, NT, VS, S_NODAL>(a, s);
  // edge sums: 8 complex rows per row of the tile, so fewer rows (256 x 256 x 64,
  // FP32: 4 rows 267 us, 8 rows 378; two columns per thread 289)
  if (a.force == 4) return launch_force_3d_t<T, NX, NX >= 128 ? 4 : 8, force_threads3<NX, 1>(), 1, S_EDGE>(a, s);
  if constexpr (NX >= 64) {
    if (a.var_a == 1) return launch_force_3d_t<T, NX, TY / 2, NT, VS, S_STRAIN>(a, s);
    if constexpr (NX >= 128 && sizeof(T) == 4) {
      if (a.var_a == 2) return launch_force_3d_t<T, NX, 2 * TY, NT, VS, S_STRAIN>(a, s);
    }
    if constexpr (NX < 256 || sizeof(T) == 4) {   // else the shared memory does not hold the ring
      if (a.var_a == 3) return launch_force_3d_t<T, NX, TY, 2 * NT, VS, S_STRAIN>(a, s);
      if (a.var_a == 4) return launch_force_3d_t<T, NX, TY / 2, 2 * NT, VS, S_STRAIN>(a, s);
    }
  }
  // Short rows: 16 of them are marched as 4 (n_x = 16) or 8 steps one after the
  // other, so few blocks leave most SMs idle: 8 rows, or 4 in single steps, all
  // of whose loads are in flight at once (us, 16 rows and 4: 16^3 FP64 68, 32,
  // FP32 16.6, 11.5; 32 x 16 x 16 FP64 127, 35; 32^3 FP64 127, 63)
  if constexpr (NX < 64) {
    const int64_t rows = (int64_t)a.n[1] * a.n[2] * a.L, sms = device_sm_count();
    if (rows / TY < sms) {
      if (rows / 8 >= sms) return launch_force_3d_t<T, NX, 8, NT, VS, S_STRAIN>(a, s);
      return launch_force_3d_t<T, NX, 4, 4 * NX, VS, S_STRAIN>(a, s);
    }
  }
  return launch_force_3d_t<T, NX, TY, NT, VS, S_STRAIN>(a, s);
}
template <typename T> cudaError_t launch_force_3d(const PassArgs<T>& a, cudaStream_t s) {
  RVE_DISPATCH_N3(a.n[0], launch_force_3d_n, a, s)
}

template <typename T, int NX, int TY, int NT, int SRC>
cudaError_t launch_force_2d_t(const PassArgs<T>& a, cudaStream_t s) {
  constexpr int MB = sizeof(T) == 8 ? 1 : NT <= 64 ? 8 : NT <= 128 ? 4 : NT <= 512 ? 2 : 1;
  constexpr size_t sm = force_2d_smem<T, NX, TY, (NT > NX ? NT / NX : 1), force_comps2<SRC>()>();
  static_assert(sm <= 222 * 1024, "shared memory of the tile");
  auto k = force_2d<T, NX, TY, NT, MB, SRC>;
  static DeviceOnce attr;
  attr.run(current_device(), [&] { set_smem_attrs(k, sm); });
  return launch_pass(a.pdl, k, dim3(a.n[1] / TY, a.L), NT, sm, s, a);
}
// Threads: at most two rows in a row of steps (TY <= 2: one lane per row).
template <int NX, int TY> constexpr int force_threads2() {
  if (NX >= 256) return 256;
  if (NX >= 128) return TY > 2 ? 128 : 256;
  const int t = NX * (TY > 2 ? (NX == 64 ? 2 : 4) : 2);
  return t < 64 ? 64 : t;
}
template <typename T, int NX, int TY, int SRC> cudaError_t launch_force_2d_r(const PassArgs<T>& a, cudaStream_t s) {
  constexpr int NT0 = force_threads2<NX, TY>(), NT = NT0 > NX * TY ? NX * TY : NT0;
  return launch_force_2d_t<T, NX, TY, NT, SRC>(a, s);
}
// Default rows: 8 (FP64: 4) where that gives every SM a block, else half, else
// a quarter; one, on long rows, where every row gets an SM of its own.  A tile
// computes one row more than it owns, so fewer rows mean more work, but on small
// grids an idle SM costs more (FP64, 512 x 256, one load case: 64 blocks of 4
// rows against 128 of 2; with one row, 256 blocks, 193 us a call against 171.
// FP64, us, two rows and one: 1024 x 16 82, 61, 512 x 64 54, 44, 256 x 64 32,
// 26).  The edge sources have two complex rows per node row: at most half the
// rows.
template <typename T, int NX, int SRC> cudaError_t launch_force_2d_auto(const PassArgs<T>& a, cudaStream_t s) {
  constexpr int TY = sizeof(T) == 4 ? 8 : 4;
  const int64_t sms = device_sm_count(), rows = (int64_t)a.n[1] * a.L;
  if constexpr (force_comps2<SRC>() == 2) {
    if (rows / TY >= sms) return launch_force_2d_r<T, NX, TY, SRC>(a, s);
  }
  if constexpr (NX >= 64) {   // (at least two warps a row)
    if (rows <= sms) return launch_force_2d_r<T, NX, 1, SRC>(a, s);
  }
  if (TY == 4 || rows / (TY / 2) < sms) return launch_force_2d_r<T, NX, 2, SRC>(a, s);
  return launch_force_2d_r<T, NX, TY / 2, SRC>(a, s);
}
// Tile variants: 0 the default rows, 1 four (FP64: two), 2 sixteen (eight), 3
// eight (four) with twice the threads, 4 two rows; 5 (FP32, n_x = 512 or 1024)
// eight rows with each 32-point register FFT spread over a lane pair.
template <typename T, int NX>
cudaError_t launch_force_2d_n(const PassArgs<T>& a, cudaStream_t s) {
  constexpr int TY = sizeof(T) == 4 ? 8 : 4;
  if (a.force == 2) return launch_force_2d_auto<T, NX, S_NODAL>(a, s);
  if (a.force == 4) return launch_force_2d_auto<T, NX, S_EDGE>(a, s);
  if constexpr (sizeof(T) == 8) {
    if (a.force == 3) return launch_force_2d_auto<T, NX, S_GRAD>(a, s);
  }
  if constexpr (NX >= 64) {
    constexpr int NT = force_threads2<NX, TY>();
    if (a.var_a == 1) return launch_force_2d_r<T, NX, TY / 2, S_STRAIN>(a, s);
    if (a.var_a == 2) return launch_force_2d_t<T, NX, 2 * TY, NT, S_STRAIN>(a, s);
    if (a.var_a == 3) return launch_force_2d_t<T, NX, TY, 2 * NT, S_STRAIN>(a, s);
    if (a.var_a == 4) return launch_force_2d_r<T, NX, 2, S_STRAIN>(a, s);
    if constexpr (sizeof(T) == 4 && (NX == 512 || NX == 1024)) {
      if (a.var_a == 5) return launch_force_2d_t<T, NX, TY, 2 * FftSplit<NX>::N1 * TY, S_STRAIN>(a, s);
    }
  }
  return launch_force_2d_auto<T, NX, S_STRAIN>(a, s);
}
template <typename T> cudaError_t launch_force_2d(const PassArgs<T>& a, cudaStream_t s) {
  RVE_DISPATCH_N(a.n[0], launch_force_2d_n, a, s)
}

}  // namespace rve

// K5 (ORAS setup, Sec. IV-C): the owned rows of every dense subdomain inverse.
//
// Setup, per subdomain s with n_s unknowns:
//   1. dense local matrix  B_s = sum_{T in s} (K^T - k0^2 eps_T M^T)
//                               + sum_{surface faces F of s} z_F B^F,
//      z_F = i k0 sqrt(eps_F) on an interface face, eps_F the eps of the inside tet (first-order
//      impedance transmission condition of Eq. m1 on the artificial boundary); on an outer face
//      z_F = i k0 sqrt(eps_bg), or with face classes (waveguide ports) the global boundary's
//      coefficient of that face (open, metal = 0, port = i beta_p); the rows and columns of
//      metal edges are then those of the identity, as in the global matrix;
//   2. block sweeps without pivoting (the imaginary part of B_s is symmetric positive definite for
//      lossy media, so every leading block is nonsingular);
//   3. the owned rows of B_s^{-1} (restricted partition of unity, boolean D_s) are kept as
//      W_s [n_own][n_s] in the apply precision.
//
// B_s is complex symmetric (Eq. m2 is bilinear), and only its owned rows are kept.  So the sweep
// operator is used instead of Gauss-Jordan: sweeping pivot block K of a symmetric A,
//   A_KK <- -A_KK^-1,  A_IK <- T_I = A_IK A_KK^-1,  A_IJ <- A_IJ - T_I A_JK^T,
// keeps A symmetric, ends at -B^-1, and needs one triangle: half the products.  The unknowns not
// owned (set N) are swept first, and the entries with both indices swept in N are never needed
// again: neither by later pivots nor by the owned rows.  With m = |N| / n the products are
// 8 n^3 (1/2 - m^3/6 - (1 - m) m^2/2), 0.39 of Gauss-Jordan's 8 n^3 at m = 0.6.
//
// Layout: position p of an unknown in the elimination order (N ascending, padded with identity rows
// to a multiple of NB, then the owned ones ascending, padded alike), row-major [np][np], the entries
// p >= q of the triangle valid.  The panel of a step lies beside each matrix, k-major:
// P[q][p] = A[p][kb + q] and T = P A_KK^-1, so that the update's operands are contiguous.
#include <algorithm>
#include <vector>

#include "k_inverse.h"
#include "mw_internal.h"

namespace mwk {
namespace {

template <typename T>
struct Tr;
template <>
struct Tr<double2> {
  using S = double;
};
template <>
struct Tr<float2> {
  using S = float;
};

__device__ __forceinline__ double2 csqrt_principal(double a, double b) {
  const double r = sqrt(a * a + b * b);
  const double re = sqrt(0.5 * (r + a));
  double im = sqrt(fmax(0.0, 0.5 * (r - a)));
  if (b < 0.0) im = -im;
  return make_double2(re, im);
}

// Assembly.  Warp `slice` of a subdomain's 64 owns the rows p = slice (mod 64): it scans the tets, 32
// at a time, and adds the entries (p_m, p_n), p_m >= p_n, of its rows in tet order, then those of the
// surface faces; every entry has one owner, so no atomics and a fixed order.  One warp per
// subdomain walked the tets alone, a chain of dependent loads: 7.9 ms for the 108 subdomains
// of a 30 x 30 x 13 mesh.
// surf_tet codes: >= 0 inside tet of an interface face; -1 outer face with i k0 sqrt(eps_bg)
// when zc is null, else -1 - c for an outer face of class c with coefficient zc[c].
constexpr int kSlices = 64, kSliceWarps = 8;
template <typename T>
__global__ void __launch_bounds__(32 * kSliceWarps) local_assemble_kernel(InvBatch bt, OrasTopo tp, const double* __restrict__ Bsurf,
                                                             const double* __restrict__ KM,
                                                             const double* __restrict__ eps, double k0,
                                                             double eps_bg_re, double eps_bg_im,
                                                             const double2* __restrict__ zc, T* __restrict__ ws) {
  using Sc = typename Tr<T>::S;
  const int b = blockIdx.x, s = bt.d_sub[b];
  const int lane = threadIdx.x & 31;
  const int slice = blockIdx.y * kSliceWarps + (threadIdx.x >> 5);
  const int np = bt.d_np[b];
  const int32_t* pos = bt.d_pos + tp.dof_ptr[s];
  T* A = ws + bt.d_off[b];
  const double k0sq = k0 * k0;
  auto add = [&](int row, int col, double re, double im) {
    T* p = A + (int64_t)row * np + col;
    T v = *p;
    v.x += (Sc)re;
    v.y += (Sc)im;
    *p = v;
  };
  const int64_t t0 = tp.tet_ptr[s], t1 = tp.tet_ptr[s + 1];
  for (int64_t base = t0; base < t1; base += 32) {
    const int64_t q = base + lane;
    int p[6], mine = 0;
    int32_t tet = 0;
    if (q < t1) {
      tet = tp.tet_ids[q];
#pragma unroll
      for (int m = 0; m < 6; ++m) {
        p[m] = pos[tp.tet_loc[6 * q + m]];
        if (p[m] % kSlices == slice) mine |= 1 << m;
      }
    }
    unsigned hits = __ballot_sync(0xffffffffu, mine != 0);
    while (hits) {
      const int src = __ffs(hits) - 1;
      hits &= hits - 1;
      const int rows = __shfl_sync(0xffffffffu, mine, src);
      const int64_t t = __shfl_sync(0xffffffffu, tet, src);
      int pt[6];
#pragma unroll
      for (int m = 0; m < 6; ++m) pt[m] = __shfl_sync(0xffffffffu, p[m], src);
      for (int e = lane; e < 36; e += 32) {
        const int m = e / 6, n = e % 6;
        int pm = 0, pn = 0;
#pragma unroll
        for (int k = 0; k < 6; ++k) {
          if (k == m) pm = pt[k];
          if (k == n) pn = pt[k];
        }
        if (!(rows >> m & 1) || pm < pn) continue;
        const int pk = mw::packed6(m, n);
        const double Kv = KM[42 * t + pk], Mv = KM[42 * t + 21 + pk];
        add(pm, pn, Kv - (k0sq * eps[2 * t]) * Mv, -(k0sq * eps[2 * t + 1]) * Mv);
      }
      __syncwarp();
    }
  }
  const double2 sbg = csqrt_principal(eps_bg_re, eps_bg_im);
  const int64_t f0 = tp.surf_ptr[s], f1 = tp.surf_ptr[s + 1];
  for (int64_t base = f0; base < f1; base += 32) {
    const int64_t q = base + lane;
    int p[3], mine = 0;
    if (q < f1) {
#pragma unroll
      for (int m = 0; m < 3; ++m) {
        p[m] = pos[tp.surf_loc[3 * q + m]];
        if (p[m] % kSlices == slice) mine |= 1 << m;
      }
    }
    unsigned hits = __ballot_sync(0xffffffffu, mine != 0);
    while (hits) {
      const int src = __ffs(hits) - 1;
      hits &= hits - 1;
      const int rows = __shfl_sync(0xffffffffu, mine, src);
      int pt[3];
#pragma unroll
      for (int m = 0; m < 3; ++m) pt[m] = __shfl_sync(0xffffffffu, p[m], src);
      if (lane < 9) {
        const int m = lane / 3, n = lane % 3;
        const int pm = m == 0 ? pt[0] : m == 1 ? pt[1] : pt[2], pn = n == 0 ? pt[0] : n == 1 ? pt[1] : pt[2];
        if ((rows >> m & 1) && pm >= pn) {
          const int64_t fq = base + src;
          const int32_t it = tp.surf_tet[fq];
          const double Bv = Bsurf[6 * fq + mw::packed3(m, n)];
          if (it < 0 && zc) {
            const double2 z = zc[-1 - it];
            add(pm, pn, z.x * Bv, z.y * Bv);
          } else {
            const double2 sq = it >= 0 ? csqrt_principal(eps[2 * (int64_t)it], eps[2 * (int64_t)it + 1]) : sbg;
            // i k0 sqrt(eps) = (-k0 Im sqrt, k0 Re sqrt)
            add(pm, pn, (-k0 * sq.y) * Bv, (k0 * sq.x) * Bv);
          }
        }
      }
      __syncwarp();
    }
  }
}

// Identity on the padding positions, and on the rows and columns of metal edges.
template <typename T>
__global__ void identity_rows_kernel(InvBatch bt, OrasTopo tp, const uint8_t* __restrict__ metal, T* __restrict__ ws) {
  const int b = blockIdx.x, s = bt.d_sub[b];
  const int np = bt.d_np[b], mn = bt.d_mn[b];
  const int n = (int)(tp.dof_ptr[s + 1] - tp.dof_ptr[s]), no = (int)(tp.own_ptr[s + 1] - tp.own_ptr[s]);
  T* A = ws + bt.d_off[b];
  for (int p = threadIdx.x; p < np; p += blockDim.x)
    if ((p >= n - no && p < mn) || p >= mn + no) A[(int64_t)p * np + p] = T{1, 0};
  if (!metal) return;
  const int32_t* gd = tp.dofs + tp.dof_ptr[s];
  const int32_t* pos = bt.d_pos + tp.dof_ptr[s];
  for (int i = 0; i < n; ++i) {
    if (!metal[gd[i]]) continue;                    // uniform over the block
    const int p = pos[i];
    for (int j = threadIdx.x; j < np; j += blockDim.x)
      A[j < p ? (int64_t)p * np + j : (int64_t)j * np + p] = T{(typename Tr<T>::S)(j == p), 0};
    __syncthreads();
  }
}

template <typename T>
__device__ __forceinline__ T cmul(T a, T b) {
  return T{a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x};
}

// The pivot block of every matrix, inverted by Gauss-Jordan without pivoting into Dinv[b]; flags a
// pivot whose modulus is below 1e-6 (FP32) or 1e-14 (FP64) of the block's largest diagonal modulus.
// One block per matrix, NB / 16 squared entries per thread in registers, the pivot row and column
// double-buffered in shared memory: one barrier per pivot, whose latency bounds it.
template <typename T, int NB>
__global__ void __launch_bounds__(256) inv_diag_kernel(InvBatch bt, const T* __restrict__ ws, int kb,
                                                       T* __restrict__ Dinv, int32_t* __restrict__ status) {
  using Sc = typename Tr<T>::S;
  constexpr int R = NB / 16;
  __shared__ T row[2][NB], col[2][NB];
  __shared__ Sc dm[NB];
  const int b = blockIdx.x;
  const int np = bt.d_np[b];
  if (kb >= np) return;
  const T* A = ws + bt.d_off[b];
  const int ty = threadIdx.x / 16, tx = threadIdx.x % 16;
  T v[R][R];
#pragma unroll
  for (int a = 0; a < R; ++a)
#pragma unroll
    for (int c = 0; c < R; ++c) {
      const int i = ty + 16 * a, j = tx + 16 * c;
      v[a][c] = A[(int64_t)(kb + max(i, j)) * np + kb + min(i, j)];
      if (i == j) dm[i] = v[a][c].x * v[a][c].x + v[a][c].y * v[a][c].y;
    }
  __syncthreads();
  Sc dmax = 0;
  for (int i = 0; i < NB; ++i) dmax = dm[i] > dmax ? dm[i] : dmax;
  const Sc tiny = (sizeof(Sc) == 4 ? (Sc)1e-12 : (Sc)1e-28) * dmax;
#pragma unroll
  for (int ka = 0; ka < R; ++ka)
    for (int k16 = 0; k16 < 16; ++k16) {
      const int k = ka * 16 + k16, buf = k16 & 1;
      if (ty == k16)
#pragma unroll
        for (int c = 0; c < R; ++c) row[buf][tx + 16 * c] = v[ka][c];
      if (tx == k16)
#pragma unroll
        for (int a = 0; a < R; ++a) col[buf][ty + 16 * a] = v[a][ka];
      __syncthreads();
      const T p = row[buf][k];
      const Sc pm = p.x * p.x + p.y * p.y;
      T ip = T{0, 0};
      if (pm > tiny)
        ip = T{p.x / pm, -p.y / pm};
      else if (threadIdx.x == 0)
        atomicExch(status, 1);
      T t[R], r[R];
#pragma unroll
      for (int a = 0; a < R; ++a) {
        t[a] = cmul(col[buf][ty + 16 * a], ip);
        r[a] = row[buf][tx + 16 * a];
      }
#pragma unroll
      for (int a = 0; a < R; ++a)
#pragma unroll
        for (int c = 0; c < R; ++c) {
          const bool ik = ty + 16 * a == k, jk = tx + 16 * c == k;
          const T u = cmul(ik ? ip : t[a], r[c]);
          if (ik && jk)
            v[a][c] = ip;
          else if (ik)
            v[a][c] = u;
          else if (jk)
            v[a][c] = T{-t[a].x, -t[a].y};
          else
            v[a][c] = T{v[a][c].x - u.x, v[a][c].y - u.y};
        }
    }
  T* Dv = Dinv + (int64_t)b * NB * NB;
#pragma unroll
  for (int a = 0; a < R; ++a)
#pragma unroll
    for (int c = 0; c < R; ++c) Dv[(ty + 16 * a) * NB + tx + 16 * c] = v[a][c];
}

// One Newton step on the FP32 inverse X of a 64 x 64 pivot block: X + X (I - D X), the residual in
// compensated FP32 (the products' and the sums' rounding errors are carried along), so that X is
// right to FP32 rounding.  The rounding of X reaches every entry the block touches: without the step the
// owned rows' error is 1.2 times that of 32 x 32 pivots (which the larger block replaces, for half the
// passes over the matrix), with it 0.6 times.  Blocks of 16 columns, FP32 pipes.
__device__ __forceinline__ void two_prod_add(float& s, float& e, float a, float b) {
  const float p = a * b, pe = fmaf(a, b, -p);
  const float t = __fadd_rn(s, p), z = __fsub_rn(t, s);
  e = __fadd_rn(e, __fadd_rn(__fadd_rn(__fsub_rn(s, __fsub_rn(t, z)), __fsub_rn(p, z)), pe));
  s = t;
}
constexpr int kRefineCols = 16;
template <int NB>
__global__ void __launch_bounds__(256) inv_refine_kernel(InvBatch bt, const float2* __restrict__ ws, int kb,
                                                         const float2* __restrict__ X0, float2* __restrict__ X1) {
  static_assert(NB == 64, "one thread per row and four columns");
  extern __shared__ __align__(16) unsigned char smem_raw[];
  float2* Ds = reinterpret_cast<float2*>(smem_raw);  // [q][i] (symmetric)
  float2* Xs = Ds + NB * NB;                         // [q][j]
  float2* Rs = Xs + NB * NB;                         // [q][16]
  const int b = blockIdx.y;
  const int np = bt.d_np[b];
  if (kb >= np) return;
  const float2* A = ws + bt.d_off[b] + (int64_t)kb * np + kb;
  const float2* X = X0 + (int64_t)b * NB * NB;
  for (int e = threadIdx.x; e < NB * NB; e += 256) {
    const int i = e / NB, j = e % NB;
    if (i >= j) Ds[i * NB + j] = Ds[j * NB + i] = A[(int64_t)i * np + j];
    Xs[e] = X[e];
  }
  __syncthreads();
  const int i = threadIdx.x % NB, c0 = threadIdx.x / NB * 4, j0 = blockIdx.x * kRefineCols + c0;
  float re[4], im[4], ee[4], ei[4];
#pragma unroll
  for (int c = 0; c < 4; ++c) {
    re[c] = i == j0 + c ? -1.f : 0.f;
    im[c] = ee[c] = ei[c] = 0.f;
  }
#pragma unroll 2
  for (int q = 0; q < NB; ++q) {
    const float2 d = Ds[q * NB + i];
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      const float2 x = Xs[q * NB + j0 + c];
      two_prod_add(re[c], ee[c], d.x, x.x);
      two_prod_add(re[c], ee[c], -d.y, x.y);
      two_prod_add(im[c], ei[c], d.x, x.y);
      two_prod_add(im[c], ei[c], d.y, x.x);
    }
  }
#pragma unroll
  for (int c = 0; c < 4; ++c) Rs[i * kRefineCols + c0 + c] = make_float2(-(re[c] + ee[c]), -(im[c] + ei[c]));
  __syncthreads();
  float2 acc[4];
#pragma unroll
  for (int c = 0; c < 4; ++c) acc[c] = make_float2(0.f, 0.f);
#pragma unroll 4
  for (int q = 0; q < NB; ++q) {
    const float2 x = Xs[q * NB + i];                 // X is symmetric to rounding: enough for the correction
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      const float2 r = Rs[q * kRefineCols + c0 + c];
      acc[c].x = fmaf(x.x, r.x, fmaf(-x.y, r.y, acc[c].x));
      acc[c].y = fmaf(x.x, r.y, fmaf(x.y, r.x, acc[c].y));
    }
  }
  float2* Y = X1 + (int64_t)b * NB * NB + i * NB + j0;
#pragma unroll
  for (int c = 0; c < 4; ++c) {
    const float2 x = Xs[i * NB + j0 + c];
    Y[c] = make_float2(x.x + acc[c].x, x.y + acc[c].y);
  }
}

// The panel of pivot block kb: P and T of block I (rows i0 ..), T written back over A_IK (as A_KI^T
// above the pivot), A_KK <- -Dinv.  Swept blocks of N keep only P while N is swept, and nothing else
// needs them.
template <typename T, int NB>
__global__ void __launch_bounds__(256) inv_panel_kernel(InvBatch bt, T* __restrict__ ws, int kb,
                                                        const T* __restrict__ Dinv) {
  constexpr int R = NB / 16;
  extern __shared__ unsigned char smem_raw[];
  T* Ps = reinterpret_cast<T*>(smem_raw);           // [q][m], rows of NB + 1
  T* Ds = Ps + NB * (NB + 1);                       // [q][j]
  const int b = blockIdx.y;
  const int np = bt.d_np[b], mn = bt.d_mn[b], i0 = blockIdx.x * NB;
  if (kb >= np || i0 >= np) return;
  T* A = ws + bt.d_off[b];
  T* P = ws + bt.d_poff[b];
  T* Tb = P + (int64_t)NB * np;
  const T* Dv = Dinv + (int64_t)b * NB * NB;
  if (i0 == kb) {
    for (int e = threadIdx.x; e < NB * NB; e += 256) {
      const int i = e / NB, j = e % NB;
      const T d = Dv[e];
      A[(int64_t)(kb + i) * np + kb + j] = T{-d.x, -d.y};
    }
    return;
  }
  const bool below = i0 > kb;
  const bool need_t = below || i0 >= mn || kb >= mn;
  for (int e = threadIdx.x; e < NB * NB; e += 256) {
    const int u = e / NB, w = e % NB;               // w runs along a row of A
    if (below)
      Ps[w * (NB + 1) + u] = A[(int64_t)(i0 + u) * np + kb + w];
    else
      Ps[u * (NB + 1) + w] = A[(int64_t)(kb + u) * np + i0 + w];
    if (need_t) Ds[e] = Dv[e];
  }
  __syncthreads();
  for (int e = threadIdx.x; e < NB * NB; e += 256) {
    const int q = e / NB, m = e % NB;
    P[(int64_t)q * np + i0 + m] = Ps[q * (NB + 1) + m];
  }
  if (!need_t) return;
  const int tm = threadIdx.x % 16, tj = threadIdx.x / 16;
  T acc[R][R];                                      // [j][m]
#pragma unroll
  for (int j = 0; j < R; ++j)
#pragma unroll
    for (int m = 0; m < R; ++m) acc[j][m] = T{0, 0};
#pragma unroll 4
  for (int q = 0; q < NB; ++q) {
    T a[R], d[R];
#pragma unroll
    for (int m = 0; m < R; ++m) a[m] = Ps[q * (NB + 1) + tm + 16 * m];
#pragma unroll
    for (int j = 0; j < R; ++j) d[j] = Ds[q * NB + tj + 16 * j];
#pragma unroll
    for (int j = 0; j < R; ++j)
#pragma unroll
      for (int m = 0; m < R; ++m) {
        acc[j][m].x = fma(a[m].x, d[j].x, acc[j][m].x);
        acc[j][m].x = fma(-a[m].y, d[j].y, acc[j][m].x);
        acc[j][m].y = fma(a[m].x, d[j].y, acc[j][m].y);
        acc[j][m].y = fma(a[m].y, d[j].x, acc[j][m].y);
      }
  }
  __syncthreads();
#pragma unroll
  for (int j = 0; j < R; ++j)
#pragma unroll
    for (int m = 0; m < R; ++m) Ps[(tj + 16 * j) * (NB + 1) + tm + 16 * m] = acc[j][m];
  __syncthreads();
  for (int e = threadIdx.x; e < NB * NB; e += 256) {
    const int u = e / NB, w = e % NB;
    Tb[(int64_t)u * np + i0 + w] = Ps[u * (NB + 1) + w];
    if (below)
      A[(int64_t)(i0 + u) * np + kb + w] = Ps[w * (NB + 1) + u];
    else
      A[(int64_t)(kb + u) * np + i0 + w] = Ps[u * (NB + 1) + w];
  }
}

__device__ __forceinline__ void load_pair(const float2* p, float2& a, float2& b) {
  const float4 v = *reinterpret_cast<const float4*>(p);
  a = make_float2(v.x, v.y);
  b = make_float2(v.z, v.w);
}
__device__ __forceinline__ void load_pair(const double2* p, double2& a, double2& b) {
  a = p[0];
  b = p[1];
}
__device__ __forceinline__ void store_pair(float2* p, float2 a, float2 b) {
  *reinterpret_cast<float4*>(p) = make_float4(a.x, a.y, b.x, b.y);
}
__device__ __forceinline__ void store_pair(double2* p, double2 a, double2 b) {
  p[0] = a;
  p[1] = b;
}
__device__ __forceinline__ void cp_async16(void* s, const void* g) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(s)), "l"(g)
               : "memory");
}

// A_IJ -= T_I P_J^T on tiles of 128 x 64 entries of the triangle, 8 x 4 complex per thread.  FP32 (FP64)
// pipes bound it: 4.2 MFLOP per 98 KB of operands and 128 KB of A read and written (FP32, NB = 64),
// 8 x 4 outputs per 8 shared-memory wavefronts of a warp's 128 multiply-adds.  Operands arrive in four
// cp.async groups, the first products start on the first; two blocks per SM overlap one's loads and
// epilogue with the other's products.  The grid holds the tiles that exist: block -> matrix by the
// step's prefix sums, tile -> (I, J) in closed form.  (64 x 64 tiles of 4 x 4 over the full squares
// of the largest size, most of them empty, ran at 30 TFLOP/s.)
constexpr int kUpM = 128, kUpN = 64;
// Tiles (I, J <= min(2 I + 1, nj - 1)) with I below the given one.
__host__ __device__ __forceinline__ int64_t inv_tiles_below(int I, int nj) {
  const int64_t full = (int64_t)I * (I + 1);
  return 2 * I > nj ? full - 1 : full;              // the last row block of an odd nj has one less
}

template <typename T, int NB>
__global__ void __launch_bounds__(256, sizeof(T) == 8 ? 2 : 1) inv_update_kernel(InvBatch bt, T* __restrict__ ws, int kb,
                                                                       const int32_t* __restrict__ prefix) {
  constexpr int VEC = 16 / (int)sizeof(T);          // elements per 16-byte copy
  constexpr int G = 4, QG = NB / G;                 // copy groups, k rows of each
  extern __shared__ __align__(16) unsigned char smem_raw[];
  T* Ts = reinterpret_cast<T*>(smem_raw);           // [q][128]
  T* Ps = Ts + NB * kUpM;                           // [q][64]
  const int lane = threadIdx.x & 31;
  // largest b with prefix[b] <= blockIdx.x (32-way search, every warp alike)
  int lo = 0, hi = bt.count;
  while (hi - lo > 1) {
    const int step = (hi - lo + 31) / 32, q = lo + (lane + 1) * step;
    const unsigned le = __ballot_sync(0xffffffffu, q < hi && prefix[q] <= (int)blockIdx.x);
    const int k = __popc(le);
    hi = min(hi, lo + (k + 1) * step);
    lo += k * step;
  }
  const int b = lo;
  const int np = bt.d_np[b], mn = bt.d_mn[b];
  const int nj = (np + kUpN - 1) / kUpN;
  const int I0 = (kb < mn ? kb : mn) / kUpM;
  const int64_t idx = (int64_t)blockIdx.x - prefix[b] + inv_tiles_below(I0, nj);
  int I = (int)((sqrtf(4.f * (float)idx + 1.f) - 1.f) * 0.5f);
  while (inv_tiles_below(I + 1, nj) <= idx) ++I;
  while (inv_tiles_below(I, nj) > idx) --I;
  const int J = (int)(idx - inv_tiles_below(I, nj));
  const int m0 = I * kUpM, n0 = J * kUpN;
  const int rmin = kb < mn ? kb + NB : mn;          // rows below are swept unknowns of N
  if (m0 + kUpM <= rmin || (n0 >= kb && n0 + kUpN <= kb + NB)) return;
  T* A = ws + bt.d_off[b];
  const T* P = ws + bt.d_poff[b];
  const T* Tb = P + (int64_t)NB * np;
  constexpr int CM = kUpM / VEC, CN = kUpN / VEC;
#pragma unroll
  for (int g = 0; g < G; ++g) {
    for (int e = threadIdx.x; e < QG * (CM + CN); e += 256) {
      const int q = g * QG + e / (CM + CN), c = e % (CM + CN);
      if (c < CM) {
        if (m0 + c * VEC < np) cp_async16(Ts + q * kUpM + c * VEC, Tb + (int64_t)q * np + m0 + c * VEC);
      } else if (n0 + (c - CM) * VEC < np) {
        cp_async16(Ps + q * kUpN + (c - CM) * VEC, P + (int64_t)q * np + n0 + (c - CM) * VEC);
      }
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  }
  const int tr = threadIdx.x / 16, tc = threadIdx.x % 16;
  T acc[8][4];
#pragma unroll
  for (int i = 0; i < 8; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) acc[i][j] = T{0, 0};
#pragma unroll
  for (int g = 0; g < G; ++g) {
    if (g == 0)
      asm volatile("cp.async.wait_group 3;" ::: "memory");
    else if (g == 1)
      asm volatile("cp.async.wait_group 2;" ::: "memory");
    else if (g == 2)
      asm volatile("cp.async.wait_group 1;" ::: "memory");
    else
      asm volatile("cp.async.wait_group 0;" ::: "memory");
    __syncthreads();
#pragma unroll 2
    for (int q = g * QG; q < (g + 1) * QG; ++q) {
      T a[8], p[4];
#pragma unroll
      for (int i = 0; i < 8; i += 2) load_pair(Ts + q * kUpM + (i < 4 ? 0 : 64) + tr * 4 + i % 4, a[i], a[i + 1]);
#pragma unroll
      for (int j = 0; j < 4; j += 2) load_pair(Ps + q * kUpN + (j < 2 ? 0 : 32) + tc * 2, p[j], p[j + 1]);
#pragma unroll
      for (int i = 0; i < 8; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          acc[i][j].x = fma(a[i].x, p[j].x, acc[i][j].x);
          acc[i][j].x = fma(-a[i].y, p[j].y, acc[i][j].x);
          acc[i][j].y = fma(a[i].x, p[j].y, acc[i][j].y);
          acc[i][j].y = fma(a[i].y, p[j].x, acc[i][j].y);
        }
    }
  }
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const int row = m0 + (i < 4 ? 0 : 64) + tr * 4 + i % 4;
    if (row >= np || row < rmin || (row >= kb && row < kb + NB)) continue;
#pragma unroll
    for (int j = 0; j < 4; j += 2) {
      const int c = n0 + (j < 2 ? 0 : 32) + tc * 2;
      // pairs start at even columns and blocks at multiples of 32: a pair is inside or outside
      if (c > row || (c >= kb && c < kb + NB)) continue;
      T* p = A + (int64_t)row * np + c;
      T u, w;
      load_pair(p, u, w);
      store_pair(p, T{u.x - acc[i][j].x, u.y - acc[i][j].y}, T{w.x - acc[i][j + 1].x, w.y - acc[i][j + 1].y});
    }
  }
}

// W_s[r][k] = B_s^-1 [own row r][k], converted to the apply precision.
template <typename T, typename U>
__global__ void extract_owned_kernel(InvBatch bt, OrasTopo tp, const T* __restrict__ ws,
                                     const int64_t* __restrict__ w_off, U* __restrict__ W) {
  using Su = decltype(U{}.x);
  const int b = blockIdx.y, s = bt.d_sub[b];
  const int np = bt.d_np[b], mn = bt.d_mn[b];
  const int64_t n = tp.dof_ptr[s + 1] - tp.dof_ptr[s], nown = tp.own_ptr[s + 1] - tp.own_ptr[s];
  const int32_t* pos = bt.d_pos + tp.dof_ptr[s];
  const T* A = ws + bt.d_off[b];
  U* Ws = W + w_off[s];
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < nown * n; e += (int64_t)gridDim.x * blockDim.x) {
    const int64_t r = e / n, k = e - r * n;
    const int p = mn + (int)r, q = pos[k];
    const T v = A[(int64_t)max(p, q) * np + min(p, q)];
    Ws[e] = U{(Su)-v.x, (Su)-v.y};
  }
}

template <typename T, int NB>
void invert_all(const InvBatch& bt, T* ws, T* dinv, int32_t* status, cudaStream_t st) {
  constexpr size_t up_smem = sizeof(T) * NB * (kUpM + kUpN);
  constexpr size_t pa_smem = sizeof(T) * (NB * (NB + 1) + NB * NB);
  constexpr size_t re_smem = sizeof(T) * (2 * NB * NB + NB * kRefineCols);
  static const cudaError_t attr[2] = {
      cudaFuncSetAttribute(inv_update_kernel<T, NB>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)up_smem),
      cudaFuncSetAttribute(inv_panel_kernel<T, NB>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)pa_smem)};
  (void)attr;   // a failure shows at the launch
  for (int k = 0; k < bt.steps; ++k) {
    const int kb = k * NB;
    note_launch(2);
    inv_diag_kernel<T, NB><<<bt.count, 256, 0, st>>>(bt, ws, kb, dinv, status);
    T* d = dinv;
    if constexpr (sizeof(T) == sizeof(float2)) {
      static const cudaError_t ra =
          cudaFuncSetAttribute(inv_refine_kernel<NB>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)re_smem);
      (void)ra;
      d = dinv + (size_t)bt.count * NB * NB;
      note_launch(1);
      inv_refine_kernel<NB><<<dim3(NB / kRefineCols, bt.count), 256, re_smem, st>>>(bt, ws, kb, dinv, d);
    }
    inv_panel_kernel<T, NB><<<dim3((bt.np_max + NB - 1) / NB, bt.count), 256, pa_smem, st>>>(bt, ws, kb, d);
    if (bt.h_tiles[k] == 0) continue;
    note_launch(1);
    inv_update_kernel<T, NB><<<bt.h_tiles[k], 256, up_smem, st>>>(bt, ws, kb,
                                                                 bt.d_prefix + (size_t)k * (bt.count + 1));
  }
}

}  // namespace

int inv_block(int prec) { return prec == 0 ? kInvBlock64 : kInvBlock32; }

int64_t inv_update_tiles(int np, int mn, int kb) {
  if (kb >= np) return 0;
  const int nj = (np + kUpN - 1) / kUpN, ni = (np + kUpM - 1) / kUpM;
  return inv_tiles_below(ni, nj) - inv_tiles_below((kb < mn ? kb : mn) / kUpM, nj);
}

void oras_local_assemble(const InvBatch& bt, const OrasTopo& tp, const double* Bsurf, const double* KM,
                         const double* eps, double k0, double ebr, double ebi, const double2* zc, const uint8_t* metal,
                         int prec, void* ws, cudaStream_t s) {
  note_launch(2);
  const dim3 g(bt.count, kSlices / kSliceWarps);
  if (prec == 0) {
    local_assemble_kernel<double2>
        <<<g, 32 * kSliceWarps, 0, s>>>(bt, tp, Bsurf, KM, eps, k0, ebr, ebi, zc, (double2*)ws);
    identity_rows_kernel<double2><<<bt.count, 256, 0, s>>>(bt, tp, metal, (double2*)ws);
  } else {
    local_assemble_kernel<float2>
        <<<g, 32 * kSliceWarps, 0, s>>>(bt, tp, Bsurf, KM, eps, k0, ebr, ebi, zc, (float2*)ws);
    identity_rows_kernel<float2><<<bt.count, 256, 0, s>>>(bt, tp, metal, (float2*)ws);
  }
}

void oras_invert(const InvBatch& bt, int prec, void* ws, void* dinv, int32_t* status, cudaStream_t s) {
  if (prec == 0)
    invert_all<double2, kInvBlock64>(bt, (double2*)ws, (double2*)dinv, status, s);
  else
    invert_all<float2, kInvBlock32>(bt, (float2*)ws, (float2*)dinv, status, s);
}

void oras_extract(const InvBatch& bt, const OrasTopo& tp, int ws_prec, const void* ws, int w_prec,
                  const int64_t* w_off, void* W, cudaStream_t s) {
  note_launch(1);
  const dim3 g(256, bt.count);
  if (ws_prec == 0 && w_prec == 0)
    extract_owned_kernel<double2, double2><<<g, 256, 0, s>>>(bt, tp, (const double2*)ws, w_off, (double2*)W);
  else if (ws_prec == 0 && w_prec == 1)
    extract_owned_kernel<double2, float2><<<g, 256, 0, s>>>(bt, tp, (const double2*)ws, w_off, (float2*)W);
  else if (ws_prec == 1 && w_prec == 0)
    extract_owned_kernel<float2, double2><<<g, 256, 0, s>>>(bt, tp, (const float2*)ws, w_off, (double2*)W);
  else
    extract_owned_kernel<float2, float2><<<g, 256, 0, s>>>(bt, tp, (const float2*)ws, w_off, (float2*)W);
}
}  // namespace mwk

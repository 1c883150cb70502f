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
//   2. in-place blocked Gauss-Jordan without pivoting (the imaginary part of B_s is symmetric
//      positive definite for lossy media, so every leading block is nonsingular);
//   3. the owned rows of B_s^{-1} (restricted partition of unity, boolean D_s) are kept as
//      W_s [n_own][n_s] in the apply precision.
//
// Step k with pivot block K (32 unknowns):  R_J = A_KK^-1 A_KJ,  A_IJ <- A_IJ - A_IK R_J,  A_KJ <- R_J,
// A_IK <- -A_IK A_KK^-1,  A_KK <- A_KK^-1.  A swept row that is not owned enters nothing any more, neither
// later steps nor W_s: it is dropped, so step k updates the owned rows before K and all rows after K, and
// the whole takes 8 n^3 (1 - m / 2) flop, m the share of unknowns not owned, instead of 8 n^3.
// (B_s is complex symmetric, and block sweeps over one triangle need half of that again.  Measured: 2.2 times
// fewer products and errors no larger, but other roundings of the entries, hence other BF16 values of some of
// them: the tensor-core apply then moves by 6e-5.  Here every entry sees the same operations in the same
// order as in the plain Gauss-Jordan.)
//
// Layout: row-major [np][np], np the unknowns padded with identity rows to a multiple of 64.  The panels of a
// step lie beside each matrix, k-major: C[q][p] = A[row p of the active rows][kb + q] and R[q][j], so that the
// update's operands are contiguous.  Active rows: the owned ones before K, ascending, then those after K.
#include <algorithm>
#include <vector>

#include "k_inverse.h"
#include "mw_chain.cuh"
#include "mw_internal.h"
#include "mw_smem.h"

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
// at a time, and adds the entries of its rows in tet order, then those of the surface faces; every entry
// has one owner, so no atomics and a fixed order.  One warp per
// subdomain walked the tets alone, a chain of dependent loads: 7.9 ms for the 108 subdomains
// of a 30 x 30 x 13 mesh.
// surf_tet codes: >= 0 inside tet of an interface face; -1 outer face with i k0 sqrt(eps_bg)
// when zc is null, else -1 - c for an outer face of class c with coefficient zc[c].
constexpr int kSlices = 64, kSliceWarps = 8;
template <typename T>
__global__ void __launch_bounds__(32 * kSliceWarps) local_assemble_kernel(InvBatch bt, OrasTopo tp,
                                                             const double* __restrict__ Bsurf,
                                                             const double* __restrict__ KM,
                                                             const double* __restrict__ eps, double k0,
                                                             double eps_bg_re, double eps_bg_im,
                                                             const double2* __restrict__ zc, T* __restrict__ ws) {
  using Sc = typename Tr<T>::S;
  const int b = blockIdx.x, s = bt.d_sub[b];
  const int lane = threadIdx.x & 31;
  const int slice = blockIdx.y * kSliceWarps + (threadIdx.x >> 5);
  const int np = bt.d_np[b];
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
        p[m] = tp.tet_loc[6 * q + m];
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
        if (!(rows >> m & 1)) continue;
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
        p[m] = tp.surf_loc[3 * q + m];
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
        if (rows >> m & 1) {
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

// Identity on the padding rows, and on the rows and columns of metal edges.
template <typename T>
__global__ void identity_rows_kernel(InvBatch bt, OrasTopo tp, const uint8_t* __restrict__ metal, T* __restrict__ ws) {
  const int b = blockIdx.x, s = bt.d_sub[b];
  const int np = bt.d_np[b];
  const int n = (int)(tp.dof_ptr[s + 1] - tp.dof_ptr[s]);
  T* A = ws + bt.d_off[b];
  for (int p = n + threadIdx.x; p < np; p += blockDim.x) A[(int64_t)p * np + p] = T{1, 0};
  if (!metal) return;
  const int32_t* gd = tp.dofs + tp.dof_ptr[s];
  for (int64_t i = 0; i < n; ++i) {
    if (!metal[gd[i]]) continue;                    // uniform over the block
    for (int64_t j = threadIdx.x; j < n; j += blockDim.x) {
      const T v = T{(typename Tr<T>::S)(j == i), 0};
      A[i * np + j] = v;
      A[j * np + i] = v;
    }
    __syncthreads();
  }
}

// a b with the multiply-adds spelled out: the rounding does not hang on the compiler's choice.
template <typename T>
__device__ __forceinline__ T cmul(T a, T b) {
  return T{fma(a.x, b.x, -(a.y * b.y)), fma(a.x, b.y, a.y * b.x)};
}

constexpr int NB = kInvBlock;

// The pivot block of every matrix, inverted by Gauss-Jordan without pivoting into Dinv[b]; flags a
// pivot whose modulus is below 1e-6 (FP32) or 1e-14 (FP64) of the block's largest diagonal modulus.
// One block per matrix, 2 x 2 entries per thread in registers, the pivot row and column double-buffered in
// shared memory: one barrier per pivot, whose latency bounds it (with the block in shared memory, two
// barriers per pivot and a serial search for the largest diagonal entry: 50 us).
template <typename T>
__global__ void __launch_bounds__(256) inv_diag_kernel(InvBatch bt, const T* __restrict__ ws, int kb,
                                                       T* __restrict__ Dinv, int32_t* __restrict__ status) {
  chain_wait();
  using Sc = typename Tr<T>::S;
  constexpr int R = NB / 16;
  __shared__ T row[2][NB], col[2][NB];
  __shared__ Sc dm[NB];
  const int b = blockIdx.x;
  const int np = bt.d_np[b];
  if (kb >= bt.d_n[b]) return;
  const T* A = ws + bt.d_off[b];
  const int ty = threadIdx.x / 16, tx = threadIdx.x % 16;
  T v[R][R];
#pragma unroll
  for (int a = 0; a < R; ++a)
#pragma unroll
    for (int c = 0; c < R; ++c) {
      const int i = ty + 16 * a, j = tx + 16 * c;
      v[a][c] = A[(int64_t)(kb + i) * np + kb + j];
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
      const Sc pm = fma(p.x, p.x, p.y * p.y);
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
          if (ik && jk) {
            v[a][c] = ip;
          } else if (ik) {
            v[a][c] = cmul(r[c], ip);
          } else if (jk) {
            v[a][c] = T{-t[a].x, -t[a].y};
          } else {
            const T u = cmul(t[a], r[c]);
            v[a][c] = T{v[a][c].x - u.x, v[a][c].y - u.y};
          }
        }
    }
  T* Dv = Dinv + (int64_t)b * NB * NB;
#pragma unroll
  for (int a = 0; a < R; ++a)
#pragma unroll
    for (int c = 0; c < R; ++c) Dv[(ty + 16 * a) * NB + tx + 16 * c] = v[a][c];
}

// Row of A at position p of the active rows of the step at kb (nsw owned rows before it).
__device__ __forceinline__ int active_row(const int32_t* own, int nsw, int kb, int p) {
  return p < nsw ? own[p] : kb + NB + p - nsw;
}

// acc += a d (complex), in the order of the products: re re, -im im, re im, im re.
template <typename T>
__device__ __forceinline__ void cfma(T& acc, T a, T d) {
  acc.x = fma(a.x, d.x, acc.x);
  acc.x = fma(-a.y, d.y, acc.x);
  acc.y = fma(a.x, d.y, acc.y);
  acc.y = fma(a.y, d.x, acc.y);
}

// The panels of pivot block kb.  Blocks below `jt` take 64 columns: R_J = A_KK^-1 A_KJ into R and over A_KJ
// (and A_KK <- A_KK^-1); the others 64 active rows: A_IK into C, A_IK <- -A_IK A_KK^-1.
constexpr int kPan = 64;
template <typename T>
__global__ void __launch_bounds__(256) inv_panel_kernel(InvBatch bt, OrasTopo tp, T* __restrict__ ws, int kb, int jt,
                                                        const T* __restrict__ Dinv, const int32_t* __restrict__ nsws) {
  chain_wait();
  extern __shared__ unsigned char smem_raw[];
  T* Ps = reinterpret_cast<T*>(smem_raw);           // [q][64 + 1]
  T* Ds = Ps + NB * (kPan + 1);                     // [NB][NB]
  const int b = blockIdx.y;
  const int np = bt.d_np[b], n = bt.d_n[b];
  if (kb >= n) return;
  T* A = ws + bt.d_off[b];
  T* C = ws + bt.d_poff[b];
  T* Rp = C + (int64_t)NB * np;
  const T* Dv = Dinv + (int64_t)b * NB * NB;
  const bool rows = (int)blockIdx.x >= jt;
  const int m = threadIdx.x % kPan, g = threadIdx.x / kPan;   // 4 groups of 8 results
  T acc[NB / 4];
#pragma unroll
  for (int i = 0; i < NB / 4; ++i) acc[i] = T{0, 0};
  if (!rows) {
    const int j0 = blockIdx.x * kPan;
    if (j0 >= np) return;
    for (int e = threadIdx.x; e < NB * kPan; e += 256)
      Ps[e / kPan * (kPan + 1) + e % kPan] = A[(int64_t)(kb + e / kPan) * np + j0 + e % kPan];
    for (int e = threadIdx.x; e < NB * NB; e += 256) Ds[e] = Dv[e];
    __syncthreads();
#pragma unroll 4
    for (int k = 0; k < NB; ++k) {
      const T c = Ps[k * (kPan + 1) + m];
#pragma unroll
      for (int i = 0; i < NB / 4; ++i) {
        const T d = Ds[(g * (NB / 4) + i) * NB + k];
        acc[i].x = fma(d.x, c.x, acc[i].x);
        acc[i].x = fma(-d.y, c.y, acc[i].x);
        acc[i].y = fma(d.x, c.y, acc[i].y);
        acc[i].y = fma(d.y, c.x, acc[i].y);
      }
    }
    const int j = j0 + m;
    const bool in_k = j >= kb && j < kb + NB;
#pragma unroll
    for (int i = 0; i < NB / 4; ++i) {
      const int q = g * (NB / 4) + i;
      A[(int64_t)(kb + q) * np + j] = in_k ? Ds[q * NB + j - kb] : acc[i];
      Rp[(int64_t)q * np + j] = acc[i];
    }
    return;
  }
  const int s = bt.d_sub[b], nsw = nsws[b];
  const int32_t* own = tp.own_local + tp.own_ptr[s];
  const int count = nsw + max(0, n - kb - NB), p0 = (blockIdx.x - jt) * kPan;
  if (p0 >= count) return;
  for (int e = threadIdx.x; e < NB * kPan; e += 256) {
    const int p = e / NB, q = e % NB;
    Ps[q * (kPan + 1) + p] =
        p0 + p < count ? A[(int64_t)active_row(own, nsw, kb, p0 + p) * np + kb + q] : T{0, 0};
  }
  for (int e = threadIdx.x; e < NB * NB; e += 256) Ds[e] = Dv[e];
  __syncthreads();
#pragma unroll 4
  for (int k = 0; k < NB; ++k) {
    const T r = Ps[k * (kPan + 1) + m];
#pragma unroll
    for (int i = 0; i < NB / 4; ++i) cfma(acc[i], r, Ds[k * NB + g * (NB / 4) + i]);
  }
  for (int e = threadIdx.x; e < NB * kPan; e += 256)
    if (p0 + e % kPan < np) C[(int64_t)(e / kPan) * np + p0 + e % kPan] = Ps[e / kPan * (kPan + 1) + e % kPan];
  __syncthreads();
#pragma unroll
  for (int i = 0; i < NB / 4; ++i) Ps[(g * (NB / 4) + i) * (kPan + 1) + m] = T{-acc[i].x, -acc[i].y};
  __syncthreads();
  for (int e = threadIdx.x; e < NB * kPan; e += 256) {
    const int p = e / NB, q = e % NB;
    if (p0 + p < count) A[(int64_t)active_row(own, nsw, kb, p0 + p) * np + kb + q] = Ps[q * (kPan + 1) + p];
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

// A_IJ -= C_I R_J on tiles of 64 active rows x 64 columns, 8 x 4 complex per thread.  FP32 (FP64) pipes bound
// it: 1.05 MFLOP per 32 KB of operands and 64 KB of A read and written (FP32), 8 x 4 outputs per 6 shared-memory
// loads of a warp's 128 multiply-adds.  Persistent blocks of 128 threads, three per SM (FP32), take every
// gridDim-th of the step's tiles: the next tile's operands (two buffers, cp.async) and this tile's part of A (L2
// prefetch) are on their way during the products, and the matrix of a tile is found by stepping on through the
// prefix sums.  One block per tile waited for its search, its operands and A half of the time (FMA pipe 49 %).
// (4 x 4 outputs per thread over full squares of the largest size, most of them empty: 30 TFLOP/s.)
constexpr int kUp = 64;
constexpr int kUpBlocks = 3;                        // per SM, by shared memory in FP32
template <typename T>
__global__ void __launch_bounds__(128, sizeof(T) == 8 ? kUpBlocks : 1) inv_update_kernel(
    InvBatch bt, OrasTopo tp, T* __restrict__ ws, int kb, const int32_t* __restrict__ nsws,
    const int32_t* __restrict__ prefix, int n_tiles) {
  chain_wait();
  constexpr int VEC = 16 / (int)sizeof(T);          // elements per 16-byte copy
  constexpr int CC = kUp / VEC;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ int rows[kUp];
  T* Sm = reinterpret_cast<T*>(smem_raw);           // two of {C [q][64], R [q][64]}
  struct Tile {
    int np, count, nsw, p0, n0;
    T* A;
    const T* C;
    const int32_t* own;
  };
  int b = 0;
  auto locate = [&](int t, Tile& x) {
    while (prefix[b + 1] <= t) ++b;
    const int s = bt.d_sub[b];
    x.np = bt.d_np[b];
    x.nsw = nsws[b];
    x.count = x.nsw + max(0, bt.d_n[b] - kb - NB);
    const int idx = t - prefix[b], nj = x.np / kUp;
    x.p0 = idx / nj * kUp;
    x.n0 = idx % nj * kUp;
    x.A = ws + bt.d_off[b];
    x.C = ws + bt.d_poff[b];
    x.own = tp.own_local + tp.own_ptr[s];
  };
  auto fetch = [&](const Tile& x, int buf) {
    T* Cs = Sm + (size_t)buf * 2 * NB * kUp;
    for (int e = threadIdx.x; e < NB * 2 * CC; e += 128) {
      const int q = e / (2 * CC), c = e % (2 * CC);
      if (c < CC) {
        if (x.p0 + c * VEC < x.np) cp_async16(Cs + q * kUp + c * VEC, x.C + (int64_t)q * x.np + x.p0 + c * VEC);
      } else {
        cp_async16(Cs + (NB + q) * kUp + (c - CC) * VEC, x.C + (int64_t)(NB + q) * x.np + x.n0 + (c - CC) * VEC);
      }
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  const int tr = threadIdx.x / 16, tc = threadIdx.x % 16;   // rows 4 tr + 0..3 and + 32, columns 2 tc + 0..1 and + 32
  Tile cur, nxt;
  locate(blockIdx.x, cur);
  fetch(cur, 0);
  for (int t = blockIdx.x, buf = 0; t < n_tiles; t += gridDim.x, buf ^= 1) {
    const bool more = t + (int)gridDim.x < n_tiles;
    {
      // the tile's rows, and half a row of its part of A per thread into L2
      const int p = cur.p0 + (int)threadIdx.x / 2;
      const int row = p < cur.count ? active_row(cur.own, cur.nsw, kb, p) : -1;
      if (!(threadIdx.x & 1)) rows[threadIdx.x / 2] = row;
      if (row >= 0) {
        const char* a =
            reinterpret_cast<const char*>(cur.A + (int64_t)row * cur.np + cur.n0 + (threadIdx.x & 1) * (kUp / 2));
#pragma unroll
        for (int o = 0; o < (int)sizeof(T) * kUp / 2; o += 128)
          asm volatile("prefetch.global.L2 [%0];" ::"l"(a + o));
      }
    }
    if (more) {
      locate(t + gridDim.x, nxt);
      fetch(nxt, buf ^ 1);
      asm volatile("cp.async.wait_group 1;" ::: "memory");
    } else {
      asm volatile("cp.async.wait_group 0;" ::: "memory");
    }
    __syncthreads();
    const T* Cs = Sm + (size_t)buf * 2 * NB * kUp;
    const T* Rs = Cs + NB * kUp;
    T acc[8][4];
#pragma unroll
    for (int i = 0; i < 8; ++i)
#pragma unroll
      for (int j = 0; j < 4; ++j) acc[i][j] = T{0, 0};
#pragma unroll 2
    for (int q = 0; q < NB; ++q) {
      T a[8], p[4];
#pragma unroll
      for (int i = 0; i < 8; i += 2) load_pair(Cs + q * kUp + (i < 4 ? 0 : 32) + tr * 4 + i % 4, a[i], a[i + 1]);
#pragma unroll
      for (int j = 0; j < 4; j += 2) load_pair(Rs + q * kUp + (j < 2 ? 0 : 32) + tc * 2, p[j], p[j + 1]);
#pragma unroll
      for (int i = 0; i < 8; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) cfma(acc[i][j], a[i], p[j]);
    }
    // four rows at a time: all their loads of A in flight together
#pragma unroll
    for (int h = 0; h < 8; h += 4) {
      T* Ar[4];
      T u[4][4];
      bool ok[4][2];
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const int row = rows[h * 8 + tr * 4 + i];
        Ar[i] = cur.A + (int64_t)row * cur.np + cur.n0 + tc * 2;
#pragma unroll
        for (int j = 0; j < 2; ++j) {
          const int c = cur.n0 + 32 * j + tc * 2;   // pivot blocks start at multiples of 32: the pair is inside or outside
          ok[i][j] = row >= 0 && (c < kb || c >= kb + NB);
          if (ok[i][j]) load_pair(Ar[i] + 32 * j, u[i][2 * j], u[i][2 * j + 1]);
        }
      }
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 2; ++j)
          if (ok[i][j]) {
            const T x = acc[h + i][2 * j], y = acc[h + i][2 * j + 1], v = u[i][2 * j], w = u[i][2 * j + 1];
            store_pair(Ar[i] + 32 * j, T{v.x - x.x, v.y - x.y}, T{w.x - y.x, w.y - y.y});
          }
    }
    __syncthreads();                                // this buffer is filled again in the next round
    cur = nxt;
  }
}

// W_s[r][k] = B_s^-1 [own row r][k], converted to the apply precision.
template <typename T, typename U>
__global__ void extract_owned_kernel(InvBatch bt, OrasTopo tp, const T* __restrict__ ws,
                                     const int64_t* __restrict__ w_off, U* __restrict__ W) {
  using Su = decltype(U{}.x);
  const int b = blockIdx.y, s = bt.d_sub[b];
  const int64_t np = bt.d_np[b], n = bt.d_n[b], nown = tp.own_ptr[s + 1] - tp.own_ptr[s];
  const T* A = ws + bt.d_off[b];
  U* Ws = W + w_off[s];
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < nown * n; e += (int64_t)gridDim.x * blockDim.x) {
    const int64_t r = e / n, k = e - r * n;
    const T v = A[tp.own_local[tp.own_ptr[s] + r] * np + k];
    Ws[e] = U{(Su)v.x, (Su)v.y};
  }
}

template <typename T>
void invert_all(const InvBatch& bt, const OrasTopo& tp, T* ws, T* dinv, int32_t* status, cudaStream_t st) {
  constexpr size_t up_smem = sizeof(T) * NB * 2 * kUp * 2;
  constexpr size_t pa_smem = sizeof(T) * (NB * (kPan + 1) + NB * NB);
  static SmemLimit update_limit, panel_limit;
  update_limit.raise(inv_update_kernel<T>, up_smem);
  panel_limit.raise(inv_panel_kernel<T>, pa_smem);
  for (int k = 0; k < bt.steps; ++k) {
    const int kb = k * NB, jt = (bt.np_max + kPan - 1) / kPan;
    const int32_t* nsws = bt.d_nsw + (size_t)k * bt.count;
    note_launch(2);
    launch_chained(inv_diag_kernel<T>, bt.count, 256, 0, st, bt, ws, kb, dinv, status);
    launch_chained(inv_panel_kernel<T>, dim3(2 * jt, bt.count), 256, pa_smem, st, bt, tp, ws, kb, jt, dinv, nsws);
    if (bt.h_tiles[k] == 0) continue;
    note_launch(1);
    constexpr int blocks = 152 * (sizeof(T) == 8 ? kUpBlocks : 1);
    launch_chained(inv_update_kernel<T>, std::min(bt.h_tiles[k], blocks), 128, up_smem, st, bt, tp, ws, kb, nsws,
        bt.d_prefix + (size_t)k * (bt.count + 1), bt.h_tiles[k]);
  }
}

}  // namespace

int64_t inv_update_tiles(int n, int np, int nsw, int kb) {
  if (kb >= n) return 0;
  return (int64_t)((nsw + std::max(0, n - kb - NB) + kUp - 1) / kUp) * (np / kUp);
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

void oras_invert(const InvBatch& bt, const OrasTopo& tp, int prec, void* ws, void* dinv, int32_t* status,
                 cudaStream_t s) {
  if (prec == 0)
    invert_all<double2>(bt, tp, (double2*)ws, (double2*)dinv, status, s);
  else
    invert_all<float2>(bt, tp, (float2*)ws, (float2*)dinv, status, s);
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

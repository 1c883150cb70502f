// Learned initialiser (no counterpart in the paper): forward and backward
// kernels of  x -> relu(W1 x + b1) -> relu(W2 . + b2) -> reshape 16x4^3 -> convT(16->16) -> relu
// -> convT(16->8) -> relu -> convT(8->2) -> 32^3 x 2,  convT = 3D transposed convolution with
// kernel 4, stride 2, padding 1:  out[co][o] = b[co] + sum_ci sum_k in[ci][i] w[ci][co][k],
// o = 2 i - 1 + k per axis.  W1, W2 are read as BF16, everything accumulates in FP32.  All
// reductions are deterministic (fixed per-thread order, fixed trees, no atomics).
#include <cuda_bf16.h>

#include <algorithm>

#include "k_nn.h"
#include "mw_chain.cuh"
#include "mw_internal.h"
#include "mw_smem.h"

namespace mwk {
namespace {

// Dense layers.  C[m][n] = sum_k A(m, k) B(k, n), k ascending, in tiles of TM x TN outputs, RM x RN per
// thread, K steps of 32 in two shared-memory buffers (the next step's global loads are in flight
// while one is multiplied).  A(m, k) = A[m lda + k] (AK) or A[k lda + m]; B(k, n) = B[n ldb + k] (BK) or
// B[k ldb + n], float or BF16.  Both tiles lie k-major in shared memory, so a thread's operands are
// float4s; a tile read along k is transposed on the way in, its columns XORed by their k quad so that
// neither the transposing stores nor the float4 loads meet bank conflicts.
// Split K: the CTA of blockIdx.z sums k in [z kchunk, (z + 1) kchunk) and, when P is given, writes
// its partial sums to P[z][m][n] for gemm_reduce_kernel.  Otherwise the epilogue runs here:
// v + bias[n], then max(v, 0) with relu, then 0 where mask[m][n] is not positive (a ReLU's backward).
// What bounds it: at 64 samples the tile grid is small (64 x 1024 outputs) and the FP32 pipes wait
// for operands.  64 x 64 tiles with one shared-memory load per two FMAs and no load in flight during
// the products took 73 us for 64 x 1024 x 2048 and 24 us for the 1024 x 2048 x 64 gradient.
constexpr int TK = 32;

struct GemmArgs {
  int64_t lda, ldb;
  const float* bias;
  const float* mask;
  float* C;
  float* P;
  int M, N, K, kchunk;
  bool relu, va, vb, vc;   // 16-byte loads of A and B, 16-byte stores of C / P
};

__device__ __forceinline__ void unpack_row(const float* p, float (&v)[4]) {
  const float4 q = *reinterpret_cast<const float4*>(p);
  v[0] = q.x;
  v[1] = q.y;
  v[2] = q.z;
  v[3] = q.w;
}
__device__ __forceinline__ void unpack_row(const __nv_bfloat16* p, float (&v)[8]) {
  const uint4 q = *reinterpret_cast<const uint4*>(p);
  const uint32_t u[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    v[2 * i] = __uint_as_float(u[i] << 16);
    v[2 * i + 1] = __uint_as_float(u[i] & 0xffff0000u);
  }
}

// One operand tile of R rows (m or n) x 32 k: NT threads, W = 16 bytes worth of elements per unit.
template <typename T, bool KC, int R, int NT>
struct TileIo {
  static constexpr int W = 16 / (int)sizeof(T);
  static constexpr int UPR = (KC ? TK : R) / W;                 // units along the contiguous axis
  static constexpr int UNITS = R * TK / W;
  static constexpr int PER = (UNITS + NT - 1) / NT;
  float v[PER][W];
  __device__ __forceinline__ void load(const T* __restrict__ A, int64_t ld, int r0, int rows, int k0, int kend,
                                       bool vec) {
#pragma unroll
    for (int q = 0; q < PER; ++q) {
      const int u = threadIdx.x + q * NT;
      if (UNITS % NT != 0 && u >= UNITS) break;
      const int o = u / UPR, i = u % UPR * W;                   // outer index, first inner index
      const int r = r0 + (KC ? o : i), k = k0 + (KC ? i : o);
      const int left = KC ? kend - k : rows - r;                // valid inner elements
      const bool in = KC ? r < rows : k < kend;
      const T* p = A + (KC ? (int64_t)r * ld + k : (int64_t)k * ld + r);
      if (in && vec && left >= W) {
        unpack_row(p, v[q]);
      } else {
#pragma unroll
        for (int j = 0; j < W; ++j) v[q][j] = in && j < left ? (float)p[j] : 0.f;
      }
    }
  }
  __device__ __forceinline__ void store(float* __restrict__ S) const {
#pragma unroll
    for (int q = 0; q < PER; ++q) {
      const int u = threadIdx.x + q * NT;
      if (UNITS % NT != 0 && u >= UNITS) break;
      const int o = u / UPR, i = u % UPR * W;
      if (KC) {
#pragma unroll
        for (int j = 0; j < W; ++j) S[(i + j) * R + (o ^ (((i + j) >> 2 & 7) << 2))] = v[q][j];
      } else {
#pragma unroll
        for (int j = 0; j < W; j += 4)
          *reinterpret_cast<float4*>(S + o * R + i + j) = make_float4(v[q][j], v[q][j + 1], v[q][j + 2], v[q][j + 3]);
      }
    }
  }
};

template <typename TB, bool AK, bool BK, int TM, int TN, int RM, int RN>
__global__ void __launch_bounds__((TM / RM) * (TN / RN)) gemm_kernel(const float* __restrict__ A,
                                                                     const TB* __restrict__ B, GemmArgs g) {
  chain_wait();
  constexpr int NT = (TM / RM) * (TN / RN);
  __shared__ __align__(16) float As[2][TK * TM];
  __shared__ __align__(16) float Bs[2][TK * TN];
  const int m0 = blockIdx.y * TM, n0 = blockIdx.x * TN;
  const int tr = threadIdx.x / (TN / RN) * 4, tc = threadIdx.x % (TN / RN) * 4;
  const int kbeg = blockIdx.z * g.kchunk, kend = min(g.K, kbeg + g.kchunk);
  float acc[RM][RN];
#pragma unroll
  for (int i = 0; i < RM; ++i)
#pragma unroll
    for (int j = 0; j < RN; ++j) acc[i][j] = 0.f;
  TileIo<float, AK, TM, NT> ta;
  TileIo<TB, BK, TN, NT> tb;
  ta.load(A, g.lda, m0, g.M, kbeg, kend, g.va);
  tb.load(B, g.ldb, n0, g.N, kbeg, kend, g.vb);
  int buf = 0;
  for (int k0 = kbeg; k0 < kend; k0 += TK, buf ^= 1) {
    ta.store(As[buf]);
    tb.store(Bs[buf]);
    __syncthreads();
    if (k0 + TK < kend) {
      ta.load(A, g.lda, m0, g.M, k0 + TK, kend, g.va);
      tb.load(B, g.ldb, n0, g.N, k0 + TK, kend, g.vb);
    }
#pragma unroll 8
    for (int k = 0; k < TK; ++k) {
      const int x = (k >> 2 & 7) << 2;
      float a[RM], b[RN];
#pragma unroll
      for (int i = 0; i < RM; i += 4) {
        const int m = (tr + i / 4 * (TM / (RM / 4))) ^ (AK ? x : 0);
        const float4 q = *reinterpret_cast<const float4*>(&As[buf][k * TM + m]);
        a[i] = q.x, a[i + 1] = q.y, a[i + 2] = q.z, a[i + 3] = q.w;
      }
#pragma unroll
      for (int j = 0; j < RN; j += 4) {
        const int n = (tc + j / 4 * (TN / (RN / 4))) ^ (BK ? x : 0);
        const float4 q = *reinterpret_cast<const float4*>(&Bs[buf][k * TN + n]);
        b[j] = q.x, b[j + 1] = q.y, b[j + 2] = q.z, b[j + 3] = q.w;
      }
#pragma unroll
      for (int i = 0; i < RM; ++i)
#pragma unroll
        for (int j = 0; j < RN; ++j) acc[i][j] = fmaf(a[i], b[j], acc[i][j]);
    }
    // the next step fills the other buffer, last read before this step's barrier
  }
#pragma unroll
  for (int i = 0; i < RM; ++i) {
    const int gm = m0 + tr + i / 4 * (TM / (RM / 4)) + i % 4;
    if (gm >= g.M) continue;
#pragma unroll
    for (int j = 0; j < RN; j += 4) {
      const int gn = n0 + tc + j / 4 * (TN / (RN / 4));
      float v[4] = {acc[i][j], acc[i][j + 1], acc[i][j + 2], acc[i][j + 3]};
      float* out = g.P ? g.P + ((int64_t)blockIdx.z * g.M + gm) * g.N + gn : g.C + (int64_t)gm * g.N + gn;
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        if (g.P || gn + q >= g.N) continue;
        if (g.bias) v[q] += g.bias[gn + q];
        if (g.relu) v[q] = v[q] > 0.f ? v[q] : 0.f;
        if (g.mask) v[q] = g.mask[(int64_t)gm * g.N + gn + q] > 0.f ? v[q] : 0.f;
      }
      if (g.vc && gn + 4 <= g.N) {
        *reinterpret_cast<float4*>(out) = make_float4(v[0], v[1], v[2], v[3]);
      } else {
#pragma unroll
        for (int q = 0; q < 4; ++q)
          if (gn + q < g.N) out[q] = v[q];
      }
    }
  }
}

// C = sum_z P[z] (z ascending), then the epilogue of gemm_kernel.
__global__ void gemm_reduce_kernel(const float* __restrict__ P, int nz, GemmArgs g) {
  chain_wait();
  const int64_t MN = (int64_t)g.M * g.N;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < MN; i += (int64_t)gridDim.x * blockDim.x) {
    float v = 0.f;
#pragma unroll 8
    for (int z = 0; z < nz; ++z) v += P[z * MN + i];
    if (g.bias) v += g.bias[i % g.N];
    if (g.relu) v = v > 0.f ? v : 0.f;
    if (g.mask) v = g.mask[i] > 0.f ? v : 0.f;
    g.C[i] = v;
  }
}

// The transposed convolutions: D = 4, 8, 16 input positions per axis, Do = 2 D.  All three are
// bound by operand delivery to the FP32 pipes (about 19 MFLOP per sample and direction, activations
// and weights in L1 / L2 / shared memory): the earlier forms issued one to two loads per FMA (a tap's
// weight and value each) and ran at 3.6 TFLOP/s.  Here a thread owns a pair of neighbouring
// positions and several channels, reads its neighbourhood once per channel with wide loads and a
// quadruple of taps per shared-memory load, so one load feeds four to eight FMAs.  Every sum runs in
// the order stated at its kernel; taps outside the volume are skipped, not multiplied by zero.
//
// Forward.  Output o = 2 j + p of cell j takes input j + d with tap k = p + 1 - 2 d (d = -1, 0, 1):
// a thread computes the 2 x 8 outputs of cells (jz, jy, jx), (jz, jy, jx + 1) for COG channels from
// 3 x 3 x 4 inputs.  Walking d = +1, 0, -1 along z, then y, then x takes the taps of every output in
// ascending order: per output the sum runs over ci, then kz, ky, kx ascending.
constexpr int kConvThreads = 128;
constexpr int kConvCog = 2;   // output channels per thread (forward): measured equal to 4, more blocks
template <int D, int CI, int CO, bool RELU>
__global__ void __launch_bounds__(kConvThreads) convT_fwd_kernel(const float* __restrict__ x,
                                                                 const float* __restrict__ w,
                                                                 const float* __restrict__ bias,
                                                                 float* __restrict__ y, int B) {
  chain_wait();
  constexpr int COG = kConvCog, DD = 2 * D;
  __shared__ float4 sw[CI * COG * 16];              // [ci][co][kz][ky] of kx quadruples
  const int co0 = blockIdx.y * COG;
  for (int q = threadIdx.x; q < CI * COG * 16; q += kConvThreads)
    sw[q] = reinterpret_cast<const float4*>(w)[(q / (COG * 16) * CO + co0) * 16 + q % (COG * 16)];
  __syncthreads();
  const int64_t t = (int64_t)blockIdx.x * kConvThreads + threadIdx.x;
  if (t >= (int64_t)B * D * D * (D / 2)) return;
  const int jx = 2 * (int)(t % (D / 2)), jy = (int)(t / (D / 2) % D), jz = (int)(t / (D / 2 * D) % D);
  const int64_t bb = t / (D / 2 * D * D);
  const bool lo[3] = {jx > 0, jy > 0, jz > 0}, hi[3] = {jx + 2 < D, jy + 1 < D, jz + 1 < D};
  float acc[COG][2][2][2][2];                       // [co][pz][py][cell][px]
#pragma unroll
  for (int co = 0; co < COG; ++co)
#pragma unroll
    for (int q = 0; q < 16; ++q) acc[co][q >> 3][(q >> 2) & 1][(q >> 1) & 1][q & 1] = bias[co0 + co];
  const float* xc = x + (bb * CI * D + jz) * D * D + jy * D + jx;
  auto load = [&](float (&v)[3][3][4]) {
#pragma unroll
    for (int a = 0; a < 3; ++a)
#pragma unroll
      for (int e = 0; e < 3; ++e) {
        const bool ok = (a == 1 || (a == 0 ? lo[2] : hi[2])) && (e == 1 || (e == 0 ? lo[1] : hi[1]));
        const float* r = xc + (a - 1) * D * D + (e - 1) * D;
        const float2 m = ok ? *reinterpret_cast<const float2*>(r) : make_float2(0.f, 0.f);
        v[a][e][0] = ok && lo[0] ? r[-1] : 0.f;
        v[a][e][1] = m.x;
        v[a][e][2] = m.y;
        v[a][e][3] = ok && hi[0] ? r[2] : 0.f;
      }
  };
  float nx[3][3][4];
  if (D < 16) load(nx);
  for (int ci = 0; ci < CI; ++ci) {
    float xv[3][3][4];
    if (D < 16) {
      // few warps per SM: the next channel's loads are in flight during this one's products
#pragma unroll
      for (int q = 0; q < 36; ++q) xv[q / 12][q / 4 % 3][q & 3] = nx[q / 12][q / 4 % 3][q & 3];
      xc += D * D * D;
      if (ci + 1 < CI) load(nx);
    } else {
      load(xv);
      xc += D * D * D;
    }
#pragma unroll
    for (int a = 2; a >= 0; --a) {
      if (!(a == 1 || (a == 0 ? lo[2] : hi[2]))) continue;
#pragma unroll
      for (int e = 2; e >= 0; --e) {
        if (!(e == 1 || (e == 0 ? lo[1] : hi[1]))) continue;
#pragma unroll
        for (int pz = 0; pz < 2; ++pz) {
          const int kz = pz + 3 - 2 * a;
          if (kz < 0 || kz > 3) continue;
#pragma unroll
          for (int py = 0; py < 2; ++py) {
            const int ky = py + 3 - 2 * e;
            if (ky < 0 || ky > 3) continue;
#pragma unroll
            for (int co = 0; co < COG; ++co) {
              const float4 w4 = sw[(ci * COG + co) * 16 + kz * 4 + ky];
              float(&s)[2][2] = acc[co][pz][py];
              // even outputs take kx = 1 (d = 0), 3 (d = -1); odd ones kx = 0 (d = 1), 2 (d = 0)
              s[0][1] = fmaf(xv[a][e][2], w4.x, s[0][1]);
              if (hi[0]) s[1][1] = fmaf(xv[a][e][3], w4.x, s[1][1]);
              s[0][0] = fmaf(xv[a][e][1], w4.y, s[0][0]);
              s[1][0] = fmaf(xv[a][e][2], w4.y, s[1][0]);
              s[0][1] = fmaf(xv[a][e][1], w4.z, s[0][1]);
              s[1][1] = fmaf(xv[a][e][2], w4.z, s[1][1]);
              if (lo[0]) s[0][0] = fmaf(xv[a][e][0], w4.w, s[0][0]);
              s[1][0] = fmaf(xv[a][e][1], w4.w, s[1][0]);
            }
          }
        }
      }
    }
  }
#pragma unroll
  for (int co = 0; co < COG; ++co)
#pragma unroll
    for (int pz = 0; pz < 2; ++pz)
#pragma unroll
      for (int py = 0; py < 2; ++py) {
        float4 v = make_float4(acc[co][pz][py][0][0], acc[co][pz][py][0][1], acc[co][pz][py][1][0],
                               acc[co][pz][py][1][1]);
        if (RELU) {
          v.x = v.x > 0.f ? v.x : 0.f;
          v.y = v.y > 0.f ? v.y : 0.f;
          v.z = v.z > 0.f ? v.z : 0.f;
          v.w = v.w > 0.f ? v.w : 0.f;
        }
        float* o = y + (((bb * CO + co0 + co) * DD + 2 * jz + pz) * DD + 2 * jy + py) * DD + 2 * jx;
        *reinterpret_cast<float4*>(o) = v;
      }
}

// Backward-data: dx[b][ci][i] = sum_co sum_k w[ci][co][k] dy[b][co][2i - 1 + k], then 0 where the
// layer's input act[b][ci][i] is not positive (the ReLU before it).  A thread owns positions
// (iz, iy, ix), (iz, iy, ix + 1) and CIG channels (the group is blockIdx.y): per (co, kz, ky) six
// dy values serve 8 CIG FMAs.  Per output the sum runs over co, then kz, ky, kx ascending.
template <int D, int CI, int CO, int CIG>
__global__ void __launch_bounds__(kConvThreads) convT_bwd_data_kernel(const float* __restrict__ dy,
                                                                      const float* __restrict__ w,
                                                                      const float* __restrict__ act,
                                                                      float* __restrict__ dx, int B) {
  chain_wait();
  constexpr int DD = 2 * D;
  __shared__ float4 sw[CO * CIG * 16];              // [co][ci][kz][ky] of kx quadruples
  const int ci0 = blockIdx.y * CIG;
  for (int q = threadIdx.x; q < CO * CIG * 16; q += kConvThreads) {
    const int k = q % 16, c = q / 16 % CIG, co = q / (16 * CIG);
    sw[q] = reinterpret_cast<const float4*>(w)[((ci0 + c) * CO + co) * 16 + k];
  }
  __syncthreads();
  const int64_t t = (int64_t)blockIdx.x * kConvThreads + threadIdx.x;
  if (t >= (int64_t)B * D * D * (D / 2)) return;
  const int ix = 2 * (int)(t % (D / 2)), iy = (int)(t / (D / 2) % D), iz = (int)(t / (D / 2 * D) % D);
  const int64_t bb = t / (D / 2 * D * D);
  const bool xlo = ix > 0, xhi = ix + 2 < D;
  float acc[CIG][2];
#pragma unroll
  for (int c = 0; c < CIG; ++c) acc[c][0] = acc[c][1] = 0.f;
  const float* yb = dy + bb * CO * DD * DD * DD + 2 * ix;
  // the 4 x 6 values of channel and plane it = 4 co + kz
  auto load = [&](int it, float (&v)[4][6]) {
    const int oz = 2 * iz - 1 + (it & 3);
    const bool okz = oz >= 0 && oz < DD;
    const float* yz = yb + ((it >> 2) * DD + oz) * DD * DD;
#pragma unroll
    for (int ky = 0; ky < 4; ++ky) {
      const int oy = 2 * iy - 1 + ky;
      const bool ok = okz && oy >= 0 && oy < DD;
      const float* r = yz + oy * DD;
      const float4 m = ok ? *reinterpret_cast<const float4*>(r) : make_float4(0.f, 0.f, 0.f, 0.f);
      v[ky][0] = ok && xlo ? r[-1] : 0.f;
      v[ky][1] = m.x;
      v[ky][2] = m.y;
      v[ky][3] = m.z;
      v[ky][4] = m.w;
      v[ky][5] = ok && xhi ? r[4] : 0.f;
    }
  };
  float ny[4][6];
  load(0, ny);
  for (int it = 0; it < 4 * CO; ++it) {
    float yv[4][6];
#pragma unroll
    for (int q = 0; q < 24; ++q) yv[q / 6][q % 6] = ny[q / 6][q % 6];
    if (it + 1 < 4 * CO) load(it + 1, ny);          // in flight during this plane's products
    const int oz = 2 * iz - 1 + (it & 3);
    if (oz < 0 || oz >= DD) continue;
    const float4* wk = sw + (it >> 2) * CIG * 16 + (it & 3) * 4;
#pragma unroll
    for (int ky = 0; ky < 4; ++ky) {
      const int oy = 2 * iy - 1 + ky;
      if (oy < 0 || oy >= DD) continue;
#pragma unroll
      for (int c = 0; c < CIG; ++c) {
        const float4 w4 = wk[c * 16 + ky];
        if (xlo) acc[c][0] = fmaf(yv[ky][0], w4.x, acc[c][0]);
        acc[c][1] = fmaf(yv[ky][2], w4.x, acc[c][1]);
        acc[c][0] = fmaf(yv[ky][1], w4.y, acc[c][0]);
        acc[c][1] = fmaf(yv[ky][3], w4.y, acc[c][1]);
        acc[c][0] = fmaf(yv[ky][2], w4.z, acc[c][0]);
        acc[c][1] = fmaf(yv[ky][4], w4.z, acc[c][1]);
        acc[c][0] = fmaf(yv[ky][3], w4.w, acc[c][0]);
        if (xhi) acc[c][1] = fmaf(yv[ky][5], w4.w, acc[c][1]);
      }
    }
  }
#pragma unroll
  for (int c = 0; c < CIG; ++c) {
    const int64_t o = (((bb * CI + ci0 + c) * D + iz) * D + iy) * D + ix;
    const float2 m = *reinterpret_cast<const float2*>(act + o);
    *reinterpret_cast<float2*>(dx + o) = make_float2(m.x > 0.f ? acc[c][0] : 0.f, m.y > 0.f ? acc[c][1] : 0.f);
  }
}

// Backward-weights, dW[ci][co][k] = sum_b sum_i x[b][ci][i] dy[b][co][2i - 1 + k], in two
// fixed-order passes.  Pass 1: block (4 channels ci, co, kz; chunk) walks its chunk of the B D^3
// input positions for the 16 taps of one kz plane; thread t takes positions t, t + 256, ... and keeps
// the 4 x 16 tap sums in registers, so a position's 16 dy values (three loads per ky) serve 64 FMAs,
// with the next position's loads in flight; the block then sums the 256 threads' values tap by tap
// (thread order, through shared memory) into part[chunk][ci][co][k].  The blocks beyond the last chunk
// take the bias: block (co, b) writes the tree sum of dy[b][co] to bpart[co][b].  Pass 2
// (nn_final_sums_kernel) sums the chunks and the samples in order.
constexpr int kBwdWThreads = 256;
constexpr int kBwdWCi = 4;
constexpr size_t kBwdWSmem = sizeof(float) * kBwdWThreads * (kBwdWCi * 16 + 1);
template <int D, int CI, int CO>
__global__ void __launch_bounds__(kBwdWThreads) convT_bwd_w_kernel(const float* __restrict__ x,
                                                                   const float* __restrict__ dy,
                                                                   float* __restrict__ part,
                                                                   float* __restrict__ bpart, int B, int64_t chunk,
                                                                   int nchunk) {
  chain_wait();
  extern __shared__ float red[];                    // [256][65]
  constexpr int DD = 2 * D, V = D * D * D, PB = CI / kBwdWCi * CO * 4;
  if ((int)blockIdx.x >= PB * nchunk) {
    const int q = blockIdx.x - PB * nchunk, co = q % CO, b = q / CO;
    const float* yc = dy + ((int64_t)b * CO + co) * 8 * V;
    float s = 0.f;
#pragma unroll 16
    for (int v = threadIdx.x; v < 8 * V; v += kBwdWThreads) s += yc[v];
    red[threadIdx.x] = s;
    __syncthreads();
    for (int st = kBwdWThreads / 2; st > 0; st >>= 1) {
      if ((int)threadIdx.x < st) red[threadIdx.x] += red[threadIdx.x + st];
      __syncthreads();
    }
    if (threadIdx.x == 0) bpart[co * B + b] = red[0];
    return;
  }
  const int pb = blockIdx.x % PB, ch = blockIdx.x / PB;
  const int kz = pb & 3, co = (pb >> 2) % CO, ci0 = (pb >> 2) / CO * kBwdWCi;
  const int64_t total = (int64_t)B * V;
  const int64_t p0 = (int64_t)ch * chunk, p1 = min(total, p0 + chunk);
  struct Item {
    float x[kBwdWCi], y[4][4];
    bool ok, xlo, xhi, ylo, yhi;
  };
  auto load = [&](int64_t t, Item& v) {
    const int i = (int)(t % V);
    const int64_t bb = t / V;
    const int ix = i % D, iy = i / D % D, iz = i / (D * D);
    const int oz = 2 * iz - 1 + kz;
    v.ok = t < p1 && oz >= 0 && oz < DD;
    v.xlo = ix > 0, v.xhi = ix + 1 < D, v.ylo = iy > 0, v.yhi = iy + 1 < D;
#pragma unroll
    for (int c = 0; c < kBwdWCi; ++c) v.x[c] = v.ok ? x[(bb * CI + ci0 + c) * V + i] : 0.f;
    const float* yc = dy + (((bb * CO + co) * DD + oz) * DD + 2 * iy) * DD + 2 * ix;
#pragma unroll
    for (int ky = 0; ky < 4; ++ky) {
      const bool ok = v.ok && (ky != 0 || v.ylo) && (ky != 3 || v.yhi);
      const float* r = yc + (ky - 1) * DD;
      const float2 m = ok ? *reinterpret_cast<const float2*>(r) : make_float2(0.f, 0.f);
      v.y[ky][0] = ok && v.xlo ? r[-1] : 0.f;
      v.y[ky][1] = m.x;
      v.y[ky][2] = m.y;
      v.y[ky][3] = ok && v.xhi ? r[2] : 0.f;
    }
  };
  float acc[kBwdWCi][16];
#pragma unroll
  for (int k = 0; k < kBwdWCi * 16; ++k) acc[k >> 4][k & 15] = 0.f;
  Item next;
  load(p0 + threadIdx.x, next);
  for (int64_t t = p0 + threadIdx.x; t < p1; t += kBwdWThreads) {
    const Item v = next;
    load(t + kBwdWThreads, next);
    if (!v.ok) continue;
#pragma unroll
    for (int ky = 0; ky < 4; ++ky) {
      if (!((ky != 0 || v.ylo) && (ky != 3 || v.yhi))) continue;
#pragma unroll
      for (int c = 0; c < kBwdWCi; ++c) {
        if (v.xlo) acc[c][ky * 4] = fmaf(v.x[c], v.y[ky][0], acc[c][ky * 4]);
        acc[c][ky * 4 + 1] = fmaf(v.x[c], v.y[ky][1], acc[c][ky * 4 + 1]);
        acc[c][ky * 4 + 2] = fmaf(v.x[c], v.y[ky][2], acc[c][ky * 4 + 2]);
        if (v.xhi) acc[c][ky * 4 + 3] = fmaf(v.x[c], v.y[ky][3], acc[c][ky * 4 + 3]);
      }
    }
  }
  constexpr int NA = kBwdWCi * 16;
#pragma unroll
  for (int k = 0; k < NA; ++k) red[threadIdx.x * (NA + 1) + k] = acc[k >> 4][k & 15];
  __syncthreads();
  if (threadIdx.x < NA) {
    float sum = 0.f;
#pragma unroll 16
    for (int q = 0; q < kBwdWThreads; ++q) sum += red[q * (NA + 1) + threadIdx.x];
    const int c = threadIdx.x >> 4;
    part[(((int64_t)ch * CI + ci0 + c) * CO + co) * 64 + kz * 16 + (threadIdx.x & 15)] = sum;
  }
}

// Every second-pass sum of a backward pass in one launch (eight launches of 3 to 7 us before, each
// a chain of loads): output q of a segment is sum_{i < n} src[base(q) + i * stride] in i order.
struct FinalSeg {
  const float* src;
  float* dst;
  int count, n;          // outputs, terms per output
  int64_t qs, is;        // src strides of the output and of the term
};
struct FinalSums {
  FinalSeg seg[8];
  int nseg;
};
__global__ void __launch_bounds__(128) nn_final_sums_kernel(FinalSums f) {
  chain_wait();
  int q = blockIdx.x * 128 + threadIdx.x;
  for (int k = 0; k < f.nseg; ++k) {
    const FinalSeg& g = f.seg[k];
    const int span = (g.count + 127) / 128 * 128;   // a block serves one segment
    if (q >= span) {
      q -= span;
      continue;
    }
    if (q >= g.count) return;
    const float* p = g.src + q * g.qs;
    float s = 0.f;
#pragma unroll 16
    for (int i = 0; i < g.n; ++i) s += p[i * g.is];
    g.dst[q] = s;
    return;
  }
}

// MSE: dy = 2 (y - t) / n, per-block partial sums of (y - t)^2 in FP64.  Block (j, b) takes elements
// [4096 j, 4096 (j + 1)) of sample b, 16 per thread as float4s; the target of sample b is row idx[b] of t
// (b without idx), so a minibatch's targets are read where they lie.
constexpr int kMseChunk = 4096;
__global__ void __launch_bounds__(256) mse_kernel(const float* __restrict__ y, const float* __restrict__ t,
                                                  const int32_t* __restrict__ idx, int64_t width, float sc,
                                                  float* __restrict__ dy, double* __restrict__ part) {
  chain_wait();
  __shared__ double red[256];
  const int64_t b = blockIdx.y, o = (int64_t)blockIdx.x * kMseChunk + threadIdx.x * 4;
  const float* yb = y + b * width + o;
  const float* tb = t + (idx ? idx[b] : b) * width + o;
  float* db = dy + b * width + o;
  double s = 0.0;
  float4 yv[4], tv[4];
#pragma unroll
  for (int u = 0; u < 4; ++u) {
    yv[u] = *reinterpret_cast<const float4*>(yb + u * 1024);
    tv[u] = *reinterpret_cast<const float4*>(tb + u * 1024);
  }
#pragma unroll
  for (int u = 0; u < 4; ++u) {
    const float d[4] = {yv[u].x - tv[u].x, yv[u].y - tv[u].y, yv[u].z - tv[u].z, yv[u].w - tv[u].w};
    *reinterpret_cast<float4*>(db + u * 1024) = make_float4(sc * d[0], sc * d[1], sc * d[2], sc * d[3]);
#pragma unroll
    for (int q = 0; q < 4; ++q) s += (double)d[q] * d[q];
  }
  red[threadIdx.x] = s;
  __syncthreads();
  for (int st = 128; st > 0; st >>= 1) {
    if ((int)threadIdx.x < st) red[threadIdx.x] += red[threadIdx.x + st];
    __syncthreads();
  }
  if (threadIdx.x == 0) part[b * gridDim.x + blockIdx.x] = red[0];
}

__global__ void sum_parts_kernel(const double* __restrict__ part, int n, double scale, double* __restrict__ out) {
  chain_wait();
  __shared__ double red[256];
  double s = 0.0;
#pragma unroll 8
  for (int i = threadIdx.x; i < n; i += 256) s += part[i];
  red[threadIdx.x] = s;
  __syncthreads();
  for (int st = 128; st > 0; st >>= 1) {
    if ((int)threadIdx.x < st) red[threadIdx.x] += red[threadIdx.x + st];
    __syncthreads();
  }
  if (threadIdx.x == 0) *out = red[0] * scale;
}

// Adam (Kingma & Ba) with bias correction; bc1 = 1 - b1^t, bc2 = 1 - b2^t.  HBM bound: four
// parameters per thread, and the new W1 and W2 (the entries [0, n1) and [o2, o2 + n2)) leave their
// BF16 copies on the way (a pass of their own read them again before).
struct AdamArgs {
  float lr, b1, b2, eps, bc1, bc2;
  int64_t n, n1, o2, n2;
};
__device__ __forceinline__ void adam_update(float& th, float g, float& m, float& v, const AdamArgs& a) {
  // the multiply-adds are spelled out so that the rounding does not hang on the compiler's choice
  const float mi = fmaf(1.f - a.b1, g, a.b1 * m);
  const float vi = fmaf((1.f - a.b2) * g, g, a.b2 * v);
  m = mi;
  v = vi;
  th -= a.lr * (mi / a.bc1) / (sqrtf(vi / a.bc2) + a.eps);
}
__device__ __forceinline__ uint2 to_bf16x4(float4 v) {
  const __nv_bfloat162 lo = __floats2bfloat162_rn(v.x, v.y), hi = __floats2bfloat162_rn(v.z, v.w);
  return make_uint2(*reinterpret_cast<const uint32_t*>(&lo), *reinterpret_cast<const uint32_t*>(&hi));
}
__global__ void __launch_bounds__(256) adam_kernel(float* __restrict__ th, const float* __restrict__ g,
                                                   float* __restrict__ m, float* __restrict__ v,
                                                   __nv_bfloat16* __restrict__ w1, __nv_bfloat16* __restrict__ w2,
                                                   AdamArgs a) {
  chain_wait();
  const int64_t i = ((int64_t)blockIdx.x * 256 + threadIdx.x) * 4;
  if (i + 4 > a.n) {                                // the last, incomplete quadruple (all biases)
    for (int64_t k = i; k < a.n; ++k) adam_update(th[k], g[k], m[k], v[k], a);
    return;
  }
  float4 t4 = *reinterpret_cast<float4*>(th + i), m4 = *reinterpret_cast<float4*>(m + i),
         v4 = *reinterpret_cast<float4*>(v + i);
  const float4 g4 = *reinterpret_cast<const float4*>(g + i);
  adam_update(t4.x, g4.x, m4.x, v4.x, a);
  adam_update(t4.y, g4.y, m4.y, v4.y, a);
  adam_update(t4.z, g4.z, m4.z, v4.z, a);
  adam_update(t4.w, g4.w, m4.w, v4.w, a);
  *reinterpret_cast<float4*>(th + i) = t4;
  *reinterpret_cast<float4*>(m + i) = m4;
  *reinterpret_cast<float4*>(v + i) = v4;
  if (i < a.n1)
    *reinterpret_cast<uint2*>(w1 + i) = to_bf16x4(t4);
  else if (i >= a.o2 && i < a.o2 + a.n2)
    *reinterpret_cast<uint2*>(w2 + i - a.o2) = to_bf16x4(t4);
}

__global__ void to_bf16_kernel(const float* __restrict__ a, __nv_bfloat16* __restrict__ b, int64_t n) {
  chain_wait();
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
    b[i] = __float2bfloat16_rn(a[i]);
}

// dst[r] = src[idx[r]], rows of `width` floats (blockIdx.y = r).
__global__ void gather_rows_kernel(const float* __restrict__ src, const int32_t* __restrict__ idx, int64_t width,
                                   float* __restrict__ dst) {
  chain_wait();
  const float* p = src + (int64_t)idx[blockIdx.y] * width;
  float* q = dst + (int64_t)blockIdx.y * width;
  for (int64_t c = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; c < width; c += (int64_t)gridDim.x * blockDim.x)
    q[c] = p[c];
}

// Mean over the 35 points of the order-4 barycentric lattice of each tet (points
// (i v0 + j v1 + k v2 + l v3) / 4, i + j + k + l = 4) of the trilinear interpolant of a
// cell-centred [2][G][G][G] grid over box [lo, hi] (0 outside the box): an average of the grid
// over the tet.  out [T][2] += (Re, Im).
__global__ void grid_to_tets_kernel(const float* __restrict__ grid, int G, double lx, double ly, double lz, double hx,
                                    double hy, double hz, const double* __restrict__ xyz,
                                    const int32_t* __restrict__ tets, int64_t T, double* __restrict__ out) {
  chain_wait();
  const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= T) return;
  double v[4][3];
  for (int a = 0; a < 4; ++a)
    for (int d = 0; d < 3; ++d) v[a][d] = xyz[3 * (int64_t)tets[4 * t + a] + d];
  const double lo[3] = {lx, ly, lz}, hi[3] = {hx, hy, hz};
  double acc0 = 0.0, acc1 = 0.0;
  for (int i = 0; i <= 4; ++i)
    for (int j = 0; i + j <= 4; ++j)
      for (int k = 0; i + j + k <= 4; ++k) {
        const int l = 4 - i - j - k;
        double c[3];
        for (int d = 0; d < 3; ++d) c[d] = (i * v[0][d] + j * v[1][d] + k * v[2][d] + l * v[3][d]) * 0.25;
        bool in = true;
        double f[3];
        int i0[3];
        for (int d = 0; d < 3; ++d) {
          if (c[d] < lo[d] || c[d] > hi[d]) in = false;
          const double u = (c[d] - lo[d]) / (hi[d] - lo[d]) * G - 0.5;
          double fl = floor(u);
          fl = fmin(fmax(fl, 0.0), (double)(G - 2));
          i0[d] = (int)fl;
          f[d] = fmin(fmax(u - fl, 0.0), 1.0);
        }
        if (!in) continue;
        for (int dz = 0; dz < 2; ++dz)
          for (int dy = 0; dy < 2; ++dy)
            for (int dx = 0; dx < 2; ++dx) {
              const double wgt = (dz ? f[2] : 1 - f[2]) * (dy ? f[1] : 1 - f[1]) * (dx ? f[0] : 1 - f[0]);
              const int64_t cell = ((int64_t)(i0[2] + dz) * G + i0[1] + dy) * G + i0[0] + dx;
              acc0 += wgt * grid[cell];
              acc1 += wgt * grid[(int64_t)G * G * G + cell];
            }
      }
  out[2 * t] += acc0 / 35.0;
  out[2 * t + 1] += acc1 / 35.0;
}

inline int gsb(int64_t n) {
  int64_t b = (n + 255) / 256;
  return (int)(b < 152 * 16 ? (b > 0 ? b : 1) : 152 * 16);
}

}  // namespace

// K chunks of a GEMM: two CTAs per SM counted in 64 x 64 tiles, chunks of at least 256 along K in
// multiples of 16, the partials within the workspace.  The count fixes the order of the sums.
static int k_splits(int M, int N, int K, size_t ws_floats, int& kchunk) {
  const int tiles = ((N + 63) / 64) * ((M + 63) / 64);
  int z = std::max(1, std::min(K / 256, (2 * 152 + tiles - 1) / tiles));
  while (z > 1 && (size_t)z * M * N > ws_floats) --z;
  kchunk = ((K + z - 1) / z + 15) / 16 * 16;
  return (K + kchunk - 1) / kchunk;
}

template <typename TB, bool AK, bool BK, int TM, int TN, int RM, int RN>
static void gemm_launch(const float* A, const TB* B, GemmArgs g, float* ws, size_t ws_floats, cudaStream_t s) {
  const int z = k_splits(g.M, g.N, g.K, ws_floats, g.kchunk);
  auto al = [](const void* p, int64_t ld, int w) { return (uintptr_t)p % 16 == 0 && ld % w == 0; };
  g.va = al(A, g.lda, 4);
  g.vb = al(B, g.ldb, 16 / (int)sizeof(TB));
  g.P = z > 1 ? ws : nullptr;
  g.vc = al(z > 1 ? ws : g.C, g.N, 4);
  note_launch(z > 1 ? 2 : 1);
  const dim3 grid((g.N + TN - 1) / TN, (g.M + TM - 1) / TM, z);
  launch_chained(gemm_kernel<TB, AK, BK, TM, TN, RM, RN>, grid, (TM / RM) * (TN / RN), 0, s, A, B, g);
  if (z == 1) return;
  const int64_t MN = (int64_t)g.M * g.N;
  launch_chained(gemm_reduce_kernel, (int)std::min<int64_t>((MN + 255) / 256, 152 * 8), 256, 0, s, ws, z, g);
}

// 32 x 32 tiles with 4 x 4 outputs per thread where the batch is the tile's short side (512 CTAs of
// 64 threads at 64 samples and 2048 inputs), 64 x 64 with 4 x 8 for the weight gradients.
void nn_dense_fwd(const float* x, const void* W, const float* bias, float* h, int B, int N, int K, float* ws,
                  size_t ws_floats, cudaStream_t s) {
  GemmArgs g{K, K, bias, nullptr, h, nullptr, B, N, K, K, true, false, false, false};
  gemm_launch<__nv_bfloat16, true, true, 32, 32, 4, 4>(x, (const __nv_bfloat16*)W, g, ws, ws_floats, s);
}
void nn_dense_bwd_data(const float* dz, const void* W, const float* h, float* dx, int B, int N, int K, float* ws,
                       size_t ws_floats, cudaStream_t s) {
  GemmArgs g{N, K, nullptr, h, dx, nullptr, B, K, N, N, false, false, false, false};
  gemm_launch<__nv_bfloat16, true, false, 32, 32, 4, 4>(dz, (const __nv_bfloat16*)W, g, ws, ws_floats, s);
}
void nn_dense_bwd_w(const float* dz, const float* x, float* dW, int B, int N, int K, float* ws, size_t ws_floats,
                    cudaStream_t s) {
  GemmArgs g{N, K, nullptr, nullptr, dW, nullptr, N, K, B, B, false, false, false, false};
  gemm_launch<float, false, false, 64, 64, 4, 8>(dz, x, g, ws, ws_floats, s);
}
template <int D, int CI, int CO, bool RELU>
static void conv_fwd(const float* x, const float* w, const float* b, float* y, int B, cudaStream_t s) {
  const int64_t n = (int64_t)B * D * D * (D / 2);
  launch_chained(convT_fwd_kernel<D, CI, CO, RELU>, dim3((unsigned)((n + kConvThreads - 1) / kConvThreads),
      CO / kConvCog), kConvThreads, 0, s, x, w, b, y, B);
}

void nn_convT_fwd(int layer, const float* x, const float* w, const float* b, float* y, int B, cudaStream_t s) {
  note_launch(1);
  if (layer == 0)
    conv_fwd<4, 16, 16, true>(x, w, b, y, B, s);
  else if (layer == 1)
    conv_fwd<8, 16, 8, true>(x, w, b, y, B, s);
  else
    conv_fwd<16, 8, 2, false>(x, w, b, y, B, s);
}

// Chunks of the backward-weights sums of a layer: whole thread rounds, at most kConvChunks, as many as
// make Ci x Co x chunks two per SM.  The count fixes the order of the sums.
static int conv_chunks(int layer, int B, int64_t& chunk) {
  constexpr int pairs[3] = {16 * 16, 16 * 8, 8 * 2}, vox[3] = {64, 512, 4096};
  const int64_t total = (int64_t)B * vox[layer];
  int nchunk = (int)std::min<int64_t>(kConvChunks, std::max<int64_t>(1, (2 * 152 + pairs[layer] - 1) / pairs[layer]));
  chunk = (total + nchunk - 1) / nchunk;
  chunk = (chunk + kBwdWThreads - 1) / kBwdWThreads * kBwdWThreads;
  return (int)((total + chunk - 1) / chunk);
}

// CIG channels of dx per thread: fewer positions (small D) take fewer channels each, so that all
// three layers launch 16k threads or more at batch 64.
template <int LAYER, int D, int CI, int CO, int CIG>
static void conv_bwd(const float* x, const float* w, const float* dy, float* dx, int B, float* bpart, float* wpart,
                     cudaStream_t s) {
  const int64_t n = (int64_t)B * D * D * (D / 2);
  launch_chained(convT_bwd_data_kernel<D, CI, CO, CIG>, dim3((unsigned)((n + kConvThreads - 1) / kConvThreads),
      CI / CIG), kConvThreads, 0, s, dy, w, x, dx, B);
  int64_t chunk = 0;
  const int nchunk = conv_chunks(LAYER, B, chunk);
  static SmemLimit limit;
  limit.raise(convT_bwd_w_kernel<D, CI, CO>, kBwdWSmem);
  launch_chained(convT_bwd_w_kernel<D, CI, CO>, CI / kBwdWCi * CO * 4 * nchunk + CO * B, kBwdWThreads, kBwdWSmem,
      s, x, dy, wpart, bpart, B, chunk, nchunk);
}

// The partial sums of layer l start at these offsets of the bias and weight workspaces.
static int64_t bpart_off(int l, int B) { return (l == 0 ? 0 : l == 1 ? 16 : 24) * (int64_t)B; }
static int64_t wpart_off(int l) { return (int64_t)kConvChunks * 64 * (l == 0 ? 0 : l == 1 ? 256 : 384); }

void nn_convT_bwd(int layer, const float* x, const float* w, const float* dy, float* dx, int B, float* bpart,
                  float* wpart, cudaStream_t s) {
  note_launch(2);
  bpart += bpart_off(layer, B);
  wpart += wpart_off(layer);
  if (layer == 0)
    conv_bwd<0, 4, 16, 16, 2>(x, w, dy, dx, B, bpart, wpart, s);
  else if (layer == 1)
    conv_bwd<1, 8, 16, 8, 4>(x, w, dy, dx, B, bpart, wpart, s);
  else
    conv_bwd<2, 16, 8, 2, 8>(x, w, dy, dx, B, bpart, wpart, s);
}

void nn_final_sums(int B, const float* bpart, const float* wpart, float* const dw[3], float* const db[3],
                   const float* dz1, const float* dz2, int N, float* db1, float* db2, cudaStream_t s) {
  note_launch(1);
  constexpr int co[3] = {16, 8, 2}, nw[3] = {16 * 16 * 64, 16 * 8 * 64, 8 * 2 * 64};
  FinalSums f{};
  int64_t blocks = 0;
  auto add = [&](const float* src, float* dst, int count, int n, int64_t qs, int64_t is) {
    f.seg[f.nseg++] = {src, dst, count, n, qs, is};
    blocks += (count + 127) / 128;
  };
  for (int l = 0; l < 3; ++l) {
    int64_t chunk = 0;
    add(wpart + wpart_off(l), dw[l], nw[l], conv_chunks(l, B, chunk), 1, nw[l]);
    add(bpart + bpart_off(l, B), db[l], co[l], B, B, 1);
  }
  add(dz2, db2, N, B, 1, N);
  add(dz1, db1, N, B, 1, N);
  launch_chained(nn_final_sums_kernel, (unsigned)blocks, 128, 0, s, f);
}

void nn_mse(const float* y, const float* t, const int32_t* idx, int B, int64_t width, float* dy, double* part,
            double* loss, cudaStream_t s) {
  note_launch(2);
  const int64_t n = B * width;
  const int nb = (int)(width / kMseChunk);
  launch_chained(mse_kernel, dim3(nb, B), 256, 0, s, y, t, idx, width, 2.0f / (float)n, dy, part);
  launch_chained(sum_parts_kernel, 1, 256, 0, s, part, nb * B, 1.0 / (double)n, loss);
}
void nn_adam(float* th, const float* g, float* m, float* v, void* w1, void* w2, int64_t n, int64_t n1, int64_t o2,
             int64_t n2, float lr, float b1, float b2, float eps, int step, cudaStream_t s) {
  note_launch(1);
  const AdamArgs a{lr, b1, b2, eps, 1.f - powf(b1, (float)step), 1.f - powf(b2, (float)step), n, n1, o2, n2};
  launch_chained(adam_kernel, (unsigned)((n + 1023) / 1024), 256, 0, s, th, g, m, v, (__nv_bfloat16*)w1,
      (__nv_bfloat16*)w2, a);
}
void nn_to_bf16(const float* a, void* b, int64_t n, cudaStream_t s) {
  note_launch(1);
  launch_chained(to_bf16_kernel, gsb(n), 256, 0, s, a, (__nv_bfloat16*)b, n);
}
void nn_gather_rows(const float* src, const int32_t* idx, int n, int64_t width, float* dst, cudaStream_t s) {
  note_launch(1);
  launch_chained(gather_rows_kernel, dim3((unsigned)((width + 255) / 256 < 16 ? (width + 255) / 256 : 16), n),
      256, 0, s, src, idx, width, dst);
}
void nn_grid_to_tets(const float* grid, int G, const double* box, const double* xyz, const int32_t* tets, int64_t T,
                     double* out, cudaStream_t s) {
  note_launch(1);
  launch_chained(grid_to_tets_kernel, (unsigned)((T + 127) / 128), 128, 0, s, grid, G, box[0], box[1], box[2],
      box[3], box[4], box[5], xyz, tets, T, out);
}

}  // namespace mwk

// K4 on the tensor cores: z[own_s] = W_s r[dofs_s] for every subdomain s, as BF16 x BF16 -> FP32
// tcgen05 MMAs with the accumulator in tensor memory (Sec. IV-C: the subdomain solves of the
// one-level ORAS preconditioner, applied through precomputed owned-row inverses).
//
// Complex product as two real GEMMs on split planes.  W = Wr + i Wi is stored as two BF16 planes
// and the gathered input g = gr + i gi once, as B = [gr | gi] (N = 2 R_pad columns: column c
// holds gr_c, column R_pad + c holds gi_c).  Two accumulators D1 = Wr B and D2 = Wi B give
//   Re z_c = D1[c] - D2[R_pad + c],   Im z_c = D1[R_pad + c] + D2[c].
// Each complex input value is staged once (2 BF16), half the bytes of an interleaved real-GEMM
// form that needs (gr, -gi) and (gi, gr); the FLOPs and the W bytes are the same.
//
// Layouts.  All operands are K-major with the 128-byte swizzle: a tile row holds 64 BF16 of K
// (128 B, K = 64 subdomain dofs); the 16-byte chunk c of row r sits at chunk c ^ (r % 8); 8-row
// groups are 1024 B apart.  W_s is pre-tiled at setup into 128-row x 64-dof tile pairs (Wr tile,
// then Wi tile: 32 KB contiguous, in that swizzled order), so one bulk copy moves a pair into
// shared memory without a tensor map.  The gathered operand of each subdomain is written per
// apply into N x 64-dof tiles.
//
// Kernel roles (192 threads): warp 0 lane 0 issues the bulk copies, warp 1 allocates tensor
// memory and lane 0 issues the MMAs, warps 2-5 read the accumulator (tcgen05.ld) and scatter
// the owned rows.  Every mbarrier wait is bounded; on timeout the kernel records an error code,
// drains its outstanding copies (again bounded), frees tensor memory and returns.
#include <cuda_bf16.h>

#include <algorithm>
#include <mutex>
#include <string>
#include <vector>

#include "k_inverse.h"
#include "k_oras.h"
#include "k_oras_tc.h"
#include "k_mf.h"
#include "mw_async.cuh"
#include "mw_chain.cuh"
#include "mw_internal.h"
#include "mw_smem.h"

namespace mwk {
namespace {

constexpr int kTileM = 128;
constexpr int kTileKd = 64;                  // subdomain dofs (complex K) per tile
constexpr int kATileBytes = kTileM * 128;    // 16 KB
constexpr int kThreadsTc = 192;
// tcgen05 shared-memory matrix descriptor: K-major, 128-byte swizzle, 8-row groups 1024 B apart.
__device__ __forceinline__ uint64_t smem_desc(uint32_t addr) {
  uint64_t d = 0;
  d |= (uint64_t)((addr & 0x3FFFF) >> 4);        // start address
  d |= (uint64_t)1 << 16;                        // leading byte offset (unused for this layout)
  d |= (uint64_t)(1024 >> 4) << 32;              // stride byte offset
  d |= (uint64_t)1 << 46;                        // descriptor version
  d |= (uint64_t)2 << 61;                        // 128-byte swizzle
  return d;
}

// Instruction descriptor, kind::f16: D FP32, A and B BF16, both K-major, M = 128, N.
__host__ __device__ constexpr uint32_t idesc_bf16(int N) {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(128 >> 4) << 24);
}

__device__ __forceinline__ void mma_bf16(uint32_t dtmem, uint64_t adesc, uint64_t bdesc, uint32_t idesc,
                                         uint32_t accumulate) {
  asm volatile(
      "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
      " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}" ::"r"(dtmem),
      "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate)
      : "memory");
}

__device__ __forceinline__ void mma_commit(uint64_t* bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_u32(bar))
               : "memory");
}

// Eight columns of the four accumulator parts that one output value needs, with one wait.
__device__ __forceinline__ void tmem_ld8x4(uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, float (&v)[4][8]) {
  uint32_t r[32];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%32];\n"
      "tcgen05.ld.sync.aligned.32x32b.x8.b32 {%8,%9,%10,%11,%12,%13,%14,%15}, [%33];\n"
      "tcgen05.ld.sync.aligned.32x32b.x8.b32 {%16,%17,%18,%19,%20,%21,%22,%23}, [%34];\n"
      "tcgen05.ld.sync.aligned.32x32b.x8.b32 {%24,%25,%26,%27,%28,%29,%30,%31}, [%35];\n"
      "tcgen05.wait::ld.sync.aligned;"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
        "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]),
        "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]),
        "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
      : "r"(a0), "r"(a1), "r"(a2), "r"(a3)
      : "memory");
#pragma unroll
  for (int i = 0; i < 32; ++i) v[i / 8][i % 8] = __uint_as_float(r[i]);
}

// Byte offset of (row, k) in a K-major, 128-byte-swizzled tile with 64 BF16 per row.
__host__ __device__ __forceinline__ uint32_t swz(uint32_t row, uint32_t k) {
  return row * 128u + ((((k >> 3) ^ (row & 7u)) & 7u) << 4) + ((k & 7u) << 1);
}

__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi) {
  const __nv_bfloat16 a = __float2bfloat16_rn(lo), b = __float2bfloat16_rn(hi);
  return (uint32_t)__bfloat16_as_ushort(a) | ((uint32_t)__bfloat16_as_ushort(b) << 16);
}

// ---------------------------------------------------------------------------------------
// Setup: owned rows of B_s^{-1} (FP32 or FP64 workspace) -> swizzled BF16 tile pairs (Wr, Wi).
// One block per (subdomain of the batch, m tile, k tile); one 32-bit word per two dofs and plane.
// ---------------------------------------------------------------------------------------
template <typename T>
__global__ void pack_w_kernel(InvBatch bt, const int64_t* __restrict__ own_ptr, const int32_t* __restrict__ own_local,
                              const T* __restrict__ ws, const int64_t* __restrict__ sub_wtile,
                              const int32_t* __restrict__ sub_kt, uint8_t* __restrict__ W) {
  const int b = blockIdx.z;
  const int s = bt.d_sub[b];
  const int64_t n = bt.d_n[b], np = bt.d_np[b];
  const int64_t nown = own_ptr[s + 1] - own_ptr[s];
  const int mt = blockIdx.y, kt = blockIdx.x;
  const int KT = sub_kt[s];
  if (kt >= KT || (int64_t)mt * kTileM >= nown) return;
  const T* A = ws + bt.d_off[b];
  uint8_t* tr = W + ((size_t)sub_wtile[s] + ((size_t)mt * KT + kt) * 2) * kATileBytes;
  uint8_t* ti = tr + kATileBytes;
  constexpr int kPairs = kTileKd / 2;
  for (int w = threadIdx.x; w < kTileM * kPairs; w += blockDim.x) {
    const int r = w / kPairs, kp = w % kPairs;
    const int64_t q = (int64_t)mt * kTileM + r, k = (int64_t)kt * kTileKd + 2 * kp;
    float re0 = 0.f, im0 = 0.f, re1 = 0.f, im1 = 0.f;
    if (q < nown) {
      const T* row = A + (int64_t)own_local[own_ptr[s] + q] * np;
      if (k < n) {
        re0 = (float)row[k].x;
        im0 = (float)row[k].y;
      }
      if (k + 1 < n) {
        re1 = (float)row[k + 1].x;
        im1 = (float)row[k + 1].y;
      }
    }
    *reinterpret_cast<uint32_t*>(tr + swz(r, 2 * kp)) = pack_bf16(re0, re1);
    *reinterpret_cast<uint32_t*>(ti + swz(r, 2 * kp)) = pack_bf16(im0, im1);
  }
}

// The same tiles from strided FP32 blocks: output row i of the plan's "subdomain" q is row own_local[i] of the
// stack of up to two products with the same B, the rows of sign_1 A_1 (task first[q]) and then those of
// sign_2 A_2 (task second[q]; < 0: none); A_i [m_i][k] has row stride lda_i at element a_off_i of src, both
// tasks have the same k, and the signs (+1 or -1) are exact in BF16.  One block per (q, m tile, k tile).
__global__ void pack_w_stacked_kernel(const MfTask* __restrict__ tasks, const int32_t* __restrict__ first,
                                      const int32_t* __restrict__ second, const int64_t* __restrict__ own_ptr,
                                      const int32_t* __restrict__ own_local, int q0,
                                      const int64_t* __restrict__ sub_wtile, const int32_t* __restrict__ sub_kt,
                                      const float2* __restrict__ src, uint8_t* __restrict__ W) {
  const int q = q0 + (int)blockIdx.z;
  const int64_t o0 = own_ptr[q], nout = own_ptr[q + 1] - o0;
  const int mt = blockIdx.y, kt = blockIdx.x;
  const int KT = sub_kt[q];
  if (kt >= KT || (int64_t)mt * kTileM >= nout) return;
  const MfTask t1 = tasks[first[q]];
  const int j2 = second[q];
  uint8_t* tr = W + ((size_t)sub_wtile[q] + ((size_t)mt * KT + kt) * 2) * kATileBytes;
  uint8_t* ti = tr + kATileBytes;
  constexpr int kPairs = kTileKd / 2;
  for (int w = threadIdx.x; w < kTileM * kPairs; w += blockDim.x) {
    const int r = w / kPairs, kp = w % kPairs;
    const int64_t o = (int64_t)mt * kTileM + r, k = (int64_t)kt * kTileKd + 2 * kp;
    float re0 = 0.f, im0 = 0.f, re1 = 0.f, im1 = 0.f;
    if (o < nout) {
      const int64_t row = own_local[o0 + o];
      const MfTask t = row < t1.m ? t1 : tasks[j2];
      const float2* a = src + t.a_off + (row < t1.m ? row : row - t1.m) * t.lda;
      if (k < t.k) {
        re0 = t.sign * a[k].x;
        im0 = t.sign * a[k].y;
      }
      if (k + 1 < t.k) {
        re1 = t.sign * a[k + 1].x;
        im1 = t.sign * a[k + 1].y;
      }
    }
    *reinterpret_cast<uint32_t*>(tr + swz(r, 2 * kp)) = pack_bf16(re0, re1);
    *reinterpret_cast<uint32_t*>(ti + swz(r, 2 * kp)) = pack_bf16(im0, im1);
  }
}

// ---------------------------------------------------------------------------------------
// Apply, step 1: gathered operand tiles B' for every (subdomain, k tile).
// ---------------------------------------------------------------------------------------
// cscale (may be null): per-column factor of the input (a Krylov vector kept unscaled), applied
// in FP32 before the BF16 rounding.
__global__ void __launch_bounds__(128, 8) gather_b_kernel(const int32_t* __restrict__ gt_sub,
                                                       const int32_t* __restrict__ gt_kt,
                                                       const int64_t* __restrict__ dof_ptr,
                                                       const int32_t* __restrict__ dofs,
                                                       const float2* __restrict__ r, int R, int Rp,
                                                       uint8_t* __restrict__ Bt, const double* __restrict__ cscale,
                                                       int64_t ntiles, const int32_t* __restrict__ go, bool early) {
  if (early) chain_next();
  chain_wait();
  if (go && *go == 0) return;
  // Blocks of 4 warps walk the tiles with a grid stride.  Per tile (64 dofs), warp w takes dofs
  // 16w .. 16w+15 and lane c the columns c, c + 32, ...: the dof indices come in one coalesced
  // load and are handed out by shuffles, the 16 values of a lane are independent loads, and each
  // lane writes its rows c (gr) and R_pad + c (gi) as two 16-byte swizzled chunks each.  The
  // tile is then copied out with coalesced 16-byte stores.
  extern __shared__ __align__(16) uint8_t tsm[];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int N = 2 * Rp;
  const int nq = (Rp + 31) / 32;
  const int nvec16 = N * 128 / 16;
  for (int64_t g = blockIdx.x; g < ntiles; g += gridDim.x) {
    const int s = gt_sub[g], kt = gt_kt[g];
    const int64_t d0 = dof_ptr[s];
    const int64_t n = dof_ptr[s + 1] - d0;
    const int64_t k0 = (int64_t)kt * kTileKd + 16 * warp;
    const int idx = (lane < 16 && k0 + lane < n) ? dofs[d0 + k0 + lane] : -1;
    for (int q = 0; q < nq; ++q) {
      const int c = lane + 32 * q;
      float2 v[16];
#pragma unroll
      for (int jj = 0; jj < 16; ++jj) {
        const int e = __shfl_sync(0xffffffffu, idx, jj);
        v[jj] = (e >= 0 && c < R) ? r[(int64_t)e * R + c] : make_float2(0.f, 0.f);
      }
      if (c < R && cscale) {
        const float sc = (float)cscale[c];
#pragma unroll
        for (int jj = 0; jj < 16; ++jj) {
          v[jj].x *= sc;
          v[jj].y *= sc;
        }
      }
      if (c < Rp) {
        uint4 re0, re1, im0, im1;
        re0.x = pack_bf16(v[0].x, v[1].x);    re0.y = pack_bf16(v[2].x, v[3].x);
        re0.z = pack_bf16(v[4].x, v[5].x);    re0.w = pack_bf16(v[6].x, v[7].x);
        re1.x = pack_bf16(v[8].x, v[9].x);    re1.y = pack_bf16(v[10].x, v[11].x);
        re1.z = pack_bf16(v[12].x, v[13].x);  re1.w = pack_bf16(v[14].x, v[15].x);
        im0.x = pack_bf16(v[0].y, v[1].y);    im0.y = pack_bf16(v[2].y, v[3].y);
        im0.z = pack_bf16(v[4].y, v[5].y);    im0.w = pack_bf16(v[6].y, v[7].y);
        im1.x = pack_bf16(v[8].y, v[9].y);    im1.y = pack_bf16(v[10].y, v[11].y);
        im1.z = pack_bf16(v[12].y, v[13].y);  im1.w = pack_bf16(v[14].y, v[15].y);
        *reinterpret_cast<uint4*>(tsm + swz(c, 16 * warp)) = re0;
        *reinterpret_cast<uint4*>(tsm + swz(c, 16 * warp + 8)) = re1;
        *reinterpret_cast<uint4*>(tsm + swz(Rp + c, 16 * warp)) = im0;
        *reinterpret_cast<uint4*>(tsm + swz(Rp + c, 16 * warp + 8)) = im1;
      }
    }
    __syncthreads();
    uint4* tile = reinterpret_cast<uint4*>(Bt + (size_t)g * N * 128);
    for (int i = threadIdx.x; i < nvec16; i += blockDim.x) tile[i] = reinterpret_cast<const uint4*>(tsm)[i];
    __syncthreads();
  }
}

// The same tiles for the sparse sweeps, each operand row the sum of up to NS listed rows (in order, as the
// multifrontal forward sweep assembles its right-hand sides): one block per tile, a thread takes 8 rows of a
// column at a time, so a warp reads whole rows and writes one 16-byte piece per plane and row group.  Summing
// here spares the front right-hand sides a pass through memory (written, read again by the gather and, for the
// update rows, by the epilogue).
template <int NS>
__global__ void __launch_bounds__(256) gather_rows_kernel(const int32_t* __restrict__ src,
                                                          const float2* __restrict__ in,
                                                          const float2* __restrict__ arena, int R, int Rp,
                                                          uint8_t* __restrict__ Bt) {
  chain_next();
  chain_wait();
  extern __shared__ __align__(16) uint8_t tsm[];
  const int32_t* idx = src + (int64_t)blockIdx.x * kTileKd * NS;
  for (int it = threadIdx.x; it < 8 * Rp; it += blockDim.x) {
    const int c = it % Rp, g = it / Rp;
    int32_t e[8 * NS];
    const int4* ip = reinterpret_cast<const int4*>(idx + 8 * NS * g);
#pragma unroll
    for (int i = 0; i < 2 * NS; ++i) *reinterpret_cast<int4*>(e + 4 * i) = ip[i];
    float2 v[8 * NS];
#pragma unroll
    for (int i = 0; i < 8 * NS; ++i) {
      const float2* row = e[i] >= 0 ? arena + (int64_t)e[i] * R : in + (int64_t)(-2 - e[i]) * R;
      v[i] = e[i] != -1 && c < R ? row[c] : make_float2(0.f, 0.f);
    }
    float2 t[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      t[j] = v[NS * j];
#pragma unroll
      for (int q = 1; q < NS; ++q) t[j] = make_float2(t[j].x + v[NS * j + q].x, t[j].y + v[NS * j + q].y);
    }
    *reinterpret_cast<uint4*>(tsm + swz(c, 8 * g)) = make_uint4(pack_bf16(t[0].x, t[1].x), pack_bf16(t[2].x, t[3].x),
                                                                pack_bf16(t[4].x, t[5].x), pack_bf16(t[6].x, t[7].x));
    *reinterpret_cast<uint4*>(tsm + swz(Rp + c, 8 * g)) =
        make_uint4(pack_bf16(t[0].y, t[1].y), pack_bf16(t[2].y, t[3].y), pack_bf16(t[4].y, t[5].y),
                   pack_bf16(t[6].y, t[7].y));
  }
  __syncthreads();
  uint4* tile = reinterpret_cast<uint4*>(Bt + (size_t)blockIdx.x * 2 * Rp * 128);
  for (int i = threadIdx.x; i < 16 * Rp; i += blockDim.x) tile[i] = reinterpret_cast<const uint4*>(tsm)[i];
}

// ---------------------------------------------------------------------------------------
// Apply, step 2: one CTA per 128-row output tile of one subdomain.
// ---------------------------------------------------------------------------------------
struct TcArgs {
  const TcTile* tiles;
  const int32_t* own_glob;  // dense applies: row of z per output row
  const TcRow* rows;        // sparse sweeps (else null): z is the arena, z2 the result
  float2* z2;
  int z_bf16;               // z holds complex BF16 pairs (4 bytes per value) instead of float2
  int vec;                  // rows of z are whole, aligned 16-byte pieces
  const uint8_t* W;
  const uint8_t* Bt;
  float2* z;
  int R, N, stages;
  uint32_t tmem_cols;
  int32_t* err;
  const int32_t* go;        // optional: zero when the kernel starts: nothing is done
  int early;                // the gather lets this launch in when it starts
};

// Position in a ring of S stages: the stage and the parity of its current round.  Running counters: a
// remainder and a quotient by the runtime S cost the issuing thread most of the 0.23 us it spends per copy.
struct RingPos {
  int st = 0;
  uint32_t ph = 0;
  __device__ __forceinline__ void next(int S) {
    if (++st == S) {
      st = 0;
      ph ^= 1u;
    }
  }
};

// One stage: the 8-row groups of the Wr and Wi tiles and the B tile.  Whole Wr and Wi tiles are adjacent, but
// one copy of 32 KB was slower than two of 16 KB (0.7 us of 48 where the inverses come from DRAM).
__device__ __forceinline__ void copy_stage_w(uint8_t* sa, const uint8_t* w, uint32_t a_part, uint32_t b_bytes,
                                             uint64_t* bar) {
  mbar_expect_tx(bar, 2u * a_part + b_bytes);
  bulk_g2s(sa, w, a_part, bar);
  bulk_g2s(sa + kATileBytes, w + kATileBytes, a_part, bar);
}
__device__ __forceinline__ void copy_stage(uint8_t* sa, const uint8_t* w, uint32_t a_part, const uint8_t* b,
                                           uint32_t b_bytes, uint64_t* bar) {
  copy_stage_w(sa, w, a_part, b_bytes, bar);
  bulk_g2s(sa + 2u * kATileBytes, b, b_bytes, bar);
}

// The first turns of the ring.  Their copies of W start before this launch's predecessor, the gather, has completed
// (in short launches and in the sweeps it lets this launch in when it starts: 16 sparse subdomains, 15 applies of 17
// launches 15.6 -> 15.4 ms).  Nothing but the host orders these reads of W and of the tile records behind the set-up
// that wrote them: it synchronises the stream after packing W and after uploading the records.
// ring_open issues the copies and returns their count, ring_join adds the B tiles once they are there and
// leaves the position of the next turn.
__device__ __forceinline__ int ring_open(uint8_t* base, uint32_t stage_bytes, const uint8_t* Wt, uint32_t a_part,
                                         uint32_t b_bytes, int KT, int S, uint64_t* full_bar) {
  const int n = min(KT, S);
  for (int i = 0; i < n; ++i)
    copy_stage_w(base + (size_t)i * stage_bytes, Wt + (size_t)i * 2 * kATileBytes, a_part, b_bytes, &full_bar[i]);
  return n;
}
__device__ __forceinline__ RingPos ring_join(uint8_t* base, uint32_t stage_bytes, const uint8_t* Bs, uint32_t b_bytes,
                                             int n, int S, uint64_t* full_bar) {
  for (int i = 0; i < n; ++i)
    bulk_g2s(base + (size_t)i * stage_bytes + 2u * kATileBytes, Bs + (size_t)i * b_bytes, b_bytes, &full_bar[i]);
  RingPos p;
  p.st = n == S ? 0 : n;
  p.ph = n == S ? 1u : 0u;
  return p;
}

// Waits for the last copies issued: every issued copy has completed before the producer leaves.
__device__ __forceinline__ bool drain_ring(uint64_t* full_bar, RingPos p, int64_t issued, int S) {
  bool ok = true;
  if (issued < S) {
    for (int i = 0; i < (int)issued; ++i) ok &= mbar_wait(&full_bar[i], 0);
    return ok;
  }
  p.ph ^= 1u;                                       // the stage at p was last filled in the round before
  for (int i = 0; i < S; ++i, p.next(S)) ok &= mbar_wait(&full_bar[p.st], p.ph);
  return ok;
}

// Rows that the copies of a tile move: whole 8-row swizzle groups that hold owned rows.  The other rows of A
// feed only accumulator rows that the epilogue does not store.
__device__ __forceinline__ uint32_t a_part_of(const TcTile& tl) { return (uint32_t)((tl.rows + 7) / 8) * 1024u; }

// Epilogue of one accumulator row, 8 columns at a time, the next added values on their way.  A thread owns a
// whole row, so its stores are 16 bytes where the rows allow it (vec): a warp's store then touches each 32-byte
// sector twice, not four (FP32) or eight (BF16) times.
__device__ __forceinline__ TcRow epi_row(const TcArgs& a, const TcTile& tl, int row) {
  TcRow e{-1, -1, -1, -1};
  if (row < tl.rows) {
    if (a.rows) {
      const int4 t = *reinterpret_cast<const int4*>(a.rows + tl.own + row);
      e = TcRow{t.x, t.y, t.z, t.w};
    } else {
      e.out = a.own_glob[tl.own + row];
    }
  }
  return e;
}
// v[i] = z[row][cb + i], 8 columns (zero past R)
__device__ __forceinline__ void epi_load8(const TcArgs& a, int32_t row, int cb, float2 (&v)[8]) {
#pragma unroll
  for (int i = 0; i < 8; ++i) v[i] = make_float2(0.f, 0.f);
  if (row < 0) return;
  const float2* p = a.z + (int64_t)row * a.R + cb;
  if (a.vec) {
#pragma unroll
    for (int i = 0; i < 8; i += 2)
      if (cb + i < a.R) {
        const float4 t = *reinterpret_cast<const float4*>(p + i);
        v[i] = make_float2(t.x, t.y);
        v[i + 1] = make_float2(t.z, t.w);
      }
  } else {
#pragma unroll
    for (int i = 0; i < 8; ++i)
      if (cb + i < a.R) v[i] = p[i];
  }
}
struct EpiAdd {
  float2 a[8], b[8];   // the two added rows' next 8 columns
};
__device__ __forceinline__ void epi_fetch(const TcArgs& a, const TcRow& e, int cb, EpiAdd& v) {
  epi_load8(a, e.add0, cb, v.a);
  epi_load8(a, e.add1, cb, v.b);
}
__device__ __forceinline__ void epi_store(const TcArgs& a, float2* z, int32_t row, bool bf16, int cb,
                                          const float2 (&v)[8]) {
  if (row < 0) return;
  if (bf16) {
    uint32_t* zr = reinterpret_cast<uint32_t*>(z) + (int64_t)row * a.R + cb;
    if (a.vec) {
#pragma unroll
      for (int i = 0; i < 8; i += 4)
        if (cb + i < a.R)
          *reinterpret_cast<uint4*>(zr + i) =
              make_uint4(pack_bf16(v[i].x, v[i].y), pack_bf16(v[i + 1].x, v[i + 1].y),
                         pack_bf16(v[i + 2].x, v[i + 2].y), pack_bf16(v[i + 3].x, v[i + 3].y));
    } else {
#pragma unroll
      for (int i = 0; i < 8; ++i)
        if (cb + i < a.R) zr[i] = pack_bf16(v[i].x, v[i].y);
    }
    return;
  }
  float2* zr = z + (int64_t)row * a.R + cb;
  if (a.vec) {
#pragma unroll
    for (int i = 0; i < 8; i += 2)
      if (cb + i < a.R) *reinterpret_cast<float4*>(zr + i) = make_float4(v[i].x, v[i].y, v[i + 1].x, v[i + 1].y);
  } else {
#pragma unroll
    for (int i = 0; i < 8; ++i)
      if (cb + i < a.R) zr[i] = v[i];
  }
}
// The accumulator at lanes (this warp's) plus the added rows to the row's places; every lane of the warp takes
// part in the reads.
__device__ __forceinline__ void epi_tile(const TcArgs& a, uint32_t lanes, const TcRow& e, EpiAdd& nxt) {
  const int Rp = a.N / 2;
  for (int cb = 0; cb < Rp; cb += 8) {
    // Re z = D1[c] - D2[Rp + c], Im z = D1[Rp + c] + D2[c]
    float2 add[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) add[i] = make_float2(nxt.a[i].x + nxt.b[i].x, nxt.a[i].y + nxt.b[i].y);
    if (cb + 8 < Rp) epi_fetch(a, e, cb + 8, nxt);
    float d[4][8];   // Wr gr, Wr gi, Wi gr, Wi gi
    tmem_ld8x4(lanes + (uint32_t)cb, lanes + (uint32_t)(Rp + cb), lanes + (uint32_t)(a.N + cb),
               lanes + (uint32_t)(a.N + Rp + cb), d);
    float2 v[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      v[i] = make_float2(d[0][i] - d[3][i], d[1][i] + d[2][i]);
      if (e.add0 >= 0) v[i] = make_float2(v[i].x + add[i].x, v[i].y + add[i].y);
    }
    epi_store(a, a.z, e.out, a.z_bf16, cb, v);
    if (a.rows) epi_store(a, a.z2, e.z, false, cb, v);
  }
}

__global__ void __launch_bounds__(kThreadsTc, 2) oras_tc_kernel(const TcArgs a) {
  extern __shared__ uint8_t dsm[];
  __shared__ __align__(8) uint64_t full_bar[8];
  __shared__ __align__(8) uint64_t empty_bar[8];
  __shared__ __align__(8) uint64_t done_bar;
  __shared__ uint32_t tmem_base;
  __shared__ int abort_flag;
  uint8_t* base = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(dsm) + 1023) & ~(uintptr_t)1023);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int S = a.stages;
  const uint32_t b_bytes = (uint32_t)a.N * 128u;
  const uint32_t a_bytes = 2u * kATileBytes;          // Wr and Wi tiles of one k tile
  const uint32_t stage_bytes = a_bytes + b_bytes;

  if (threadIdx.x == 0) {
    for (int i = 0; i < S; ++i) {
      mbar_init(&full_bar[i], 1);
      mbar_init(&empty_bar[i], 1);
    }
    mbar_init(&done_bar, 1);
    abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_base)),
                 "r"(a.tmem_cols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = tmem_base;
  const TcTile tl = a.tiles[blockIdx.x];
  const int KT = tl.kt;
  const uint8_t* Wt = a.W + (size_t)tl.w * kATileBytes;
  const uint8_t* Bs = a.Bt + (size_t)tl.g * b_bytes;
  const uint32_t a_part = a_part_of(tl);
  int issued = 0;
  if (threadIdx.x == 0 && a.early) issued = ring_open(base, stage_bytes, Wt, a_part, b_bytes, KT, S, full_bar);
  chain_wait();
  const bool go = !a.go || *a.go != 0;

  if (!go) {
    // launched ahead of a step that is not taken: complete the copies under way
    if (threadIdx.x == 0 && issued > 0) {
      const RingPos p = ring_join(base, stage_bytes, Bs, b_bytes, issued, S, full_bar);
      if (!drain_ring(full_bar, p, issued, S)) atomicCAS(a.err, 0, 2);
    }
  } else if (warp == 0) {
    if (lane == 0) {
      // producer: bulk copies of (Wr and Wi tiles, B tile) per k tile
      RingPos p = ring_join(base, stage_bytes, Bs, b_bytes, issued, S, full_bar);
      for (int kt = issued; kt < KT; ++kt, p.next(S)) {
        if (kt >= S && !mbar_wait(&empty_bar[p.st], p.ph ^ 1u)) {
          atomicCAS(a.err, 0, 1);
          abort_flag = 1;
          break;
        }
        if (*(volatile int*)&abort_flag) break;
        copy_stage(base + (size_t)p.st * stage_bytes, Wt + (size_t)kt * a_bytes, a_part, Bs + (size_t)kt * b_bytes,
                   b_bytes, &full_bar[p.st]);
        ++issued;
      }
      // every issued copy has completed before this thread leaves
      if (!drain_ring(full_bar, p, issued, S)) atomicCAS(a.err, 0, 2);
    }
  } else if (warp == 1) {
    if (lane == 0) {
      const uint32_t idesc = idesc_bf16(a.N);
      RingPos p;
      for (int kt = 0; kt < KT; ++kt, p.next(S)) {
        const int st = p.st;
        if (!mbar_wait(&full_bar[st], p.ph)) {
          atomicCAS(a.err, 0, 3);
          abort_flag = 1;
          break;
        }
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        const uint32_t sar = smem_u32(base + (size_t)st * stage_bytes);
        const uint32_t sai = sar + kATileBytes;
        const uint32_t sb = sar + a_bytes;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          const uint32_t acc = (kt > 0 || k > 0) ? 1u : 0u;
          mma_bf16(tmem, smem_desc(sar + 32u * k), smem_desc(sb + 32u * k), idesc, acc);               // D1 = Wr B
          mma_bf16(tmem + (uint32_t)a.N, smem_desc(sai + 32u * k), smem_desc(sb + 32u * k), idesc, acc);  // D2 = Wi B
        }
        mma_commit(&empty_bar[st]);
      }
      mma_commit(&done_bar);
    }
  } else {
    // epilogue: warps 2..5 cover tensor-memory lane quadrants (warp % 4).  The output row, the C0
    // row and C0's first 8 columns are looked up while the MMAs run.
    const int quad = warp & 3;
    const TcRow e = epi_row(a, tl, quad * 32 + lane);
    EpiAdd nxt;
    epi_fetch(a, e, 0, nxt);
    bool ok = mbar_wait(&done_bar, 0);
    ok = __all_sync(0xffffffffu, ok && !*(volatile int*)&abort_flag);   // tcgen05.ld below is warp-collective
    if (!ok && lane == 0) atomicCAS(a.err, 0, 4);
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    if (ok) epi_tile(a, tmem + ((uint32_t)(quad * 32) << 16), e, nxt);
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (warp == 1) {
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(a.tmem_cols) : "memory");
  }
}

// Persistent form of oras_tc_kernel for plans of many short tiles (the sparse sweeps): the CTAs
// take the 128-row output tiles t = blockIdx.x, blockIdx.x + gridDim.x, ...; one copy ring runs
// across the CTA's tiles, and the accumulators are double-buffered in tensor memory (buffer
// i % 2 for the CTA's i-th tile), so the epilogue of one tile overlaps the copies and MMAs of
// the next.  Per tile: the same copies, MMAs in the same order and the same epilogue arithmetic
// as oras_tc_kernel, so z is bit-identical.  Waits are bounded: a wait that runs out records an
// error code and sets the abort flag, every role then stops, the producer drains its copies and
// the MMA warp waits (bounded) for its last MMAs before the accumulators are freed.
__global__ void __launch_bounds__(kThreadsTc, 2) oras_tc_persistent_kernel(const TcArgs a, int n_tiles) {
  extern __shared__ uint8_t dsm[];
  __shared__ __align__(8) uint64_t full_bar[8];
  __shared__ __align__(8) uint64_t empty_bar[8];
  __shared__ __align__(8) uint64_t acc_full[2];
  __shared__ __align__(8) uint64_t acc_empty[2];
  __shared__ __align__(8) uint64_t fin_bar;
  __shared__ uint32_t tmem_base;
  __shared__ int abort_flag;
  uint8_t* base = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(dsm) + 1023) & ~(uintptr_t)1023);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int S = a.stages;
  const uint32_t b_bytes = (uint32_t)a.N * 128u;
  const uint32_t a_bytes = 2u * kATileBytes;
  const uint32_t stage_bytes = a_bytes + b_bytes;
  volatile int* abort_v = &abort_flag;

  if (threadIdx.x == 0) {
    for (int i = 0; i < S; ++i) {
      mbar_init(&full_bar[i], 1);
      mbar_init(&empty_bar[i], 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(&acc_full[b], 1);
      mbar_init(&acc_empty[b], 4);   // one arrival per epilogue warp
    }
    mbar_init(&fin_bar, 1);
    abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_base)),
                 "r"(2u * a.tmem_cols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = tmem_base;
  TcTile tl0;           // this CTA's first tile (producer)
  int opened = 0;       // its k tiles whose W copies are under way
  if (threadIdx.x == 0) {
    tl0 = a.tiles[blockIdx.x];
    opened = ring_open(base, stage_bytes, a.W + (size_t)tl0.w * kATileBytes, a_part_of(tl0), b_bytes, tl0.kt, S,
                       full_bar);
  }
  chain_wait();

  if (warp == 0) {
    if (lane == 0) {
      int64_t it = opened;   // k tiles issued by this CTA
      RingPos p = ring_join(base, stage_bytes, a.Bt + (size_t)tl0.g * b_bytes, b_bytes, opened, S, full_bar);
      int kt = opened;
      TcTile nxt = tl0;
      for (int t = blockIdx.x; t < n_tiles && !*abort_v; t += gridDim.x, kt = 0) {
        const TcTile tl = nxt;
        if (t + (int)gridDim.x < n_tiles) nxt = a.tiles[t + gridDim.x];
        const int KT = tl.kt;
        const uint8_t* Wt = a.W + (size_t)tl.w * kATileBytes;
        const uint8_t* Bs = a.Bt + (size_t)tl.g * b_bytes;
        const uint32_t a_part = a_part_of(tl);
        for (; kt < KT; ++kt, ++it, p.next(S)) {
          if (it >= S && !mbar_wait(&empty_bar[p.st], p.ph ^ 1u)) {
            atomicCAS(a.err, 0, 11);
            *abort_v = 1;
          }
          if (*abort_v) break;
          copy_stage(base + (size_t)p.st * stage_bytes, Wt + (size_t)kt * a_bytes, a_part, Bs + (size_t)kt * b_bytes,
                     b_bytes, &full_bar[p.st]);
        }
      }
      // every issued copy has completed before this thread leaves
      if (!drain_ring(full_bar, p, it, S)) atomicCAS(a.err, 0, 12);
    }
  } else if (warp == 1) {
    if (lane == 0) {
      const uint32_t idesc = idesc_bf16(a.N);
      RingPos p;
      int i = 0;   // tiles of this CTA
      int kt_next = a.tiles[blockIdx.x].kt;
      for (int t = blockIdx.x; t < n_tiles && !*abort_v; t += gridDim.x, ++i) {
        const int KT = kt_next;
        if (t + (int)gridDim.x < n_tiles) kt_next = a.tiles[t + gridDim.x].kt;
        const int buf = i & 1;
        if (i >= 2 && !mbar_wait(&acc_empty[buf], (uint32_t)(((i >> 1) + 1) & 1))) {
          atomicCAS(a.err, 0, 13);
          *abort_v = 1;
          break;
        }
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        const uint32_t acc0 = tmem + (uint32_t)buf * a.tmem_cols;
        bool stop = false;
        for (int kt = 0; kt < KT; ++kt, p.next(S)) {
          const int st = p.st;
          if (!mbar_wait(&full_bar[st], p.ph)) {
            atomicCAS(a.err, 0, 14);
            *abort_v = 1;
            stop = true;
            break;
          }
          asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
          const uint32_t sar = smem_u32(base + (size_t)st * stage_bytes);
          const uint32_t sai = sar + kATileBytes;
          const uint32_t sb = sar + a_bytes;
#pragma unroll
          for (int k = 0; k < 4; ++k) {
            const uint32_t acc = (kt > 0 || k > 0) ? 1u : 0u;
            mma_bf16(acc0, smem_desc(sar + 32u * k), smem_desc(sb + 32u * k), idesc, acc);
            mma_bf16(acc0 + (uint32_t)a.N, smem_desc(sai + 32u * k), smem_desc(sb + 32u * k), idesc, acc);
          }
          mma_commit(&empty_bar[st]);
        }
        if (stop) break;
        mma_commit(&acc_full[buf]);
      }
      // every MMA issued by this CTA has completed before the accumulators are freed
      mma_commit(&fin_bar);
      if (!mbar_wait(&fin_bar, 0)) atomicCAS(a.err, 0, 15);
    }
  } else {
    // A tile's record is read two tiles ahead and its row numbers one tile ahead: in line, that chain of
    // dependent reads took longer than the copies of a tile with one to four k tiles (16 sparse subdomains of
    // 44x44x17 cells, 32 columns, two ring stages: a solve of 15 applies 23.9 -> 21.2 ms together with the 16-byte
    // stores).
    const int quad = warp & 3;
    const int row = quad * 32 + lane;
    const int step = gridDim.x;
    TcRow e1 = epi_row(a, a.tiles[blockIdx.x], row);
    TcTile t2;
    if ((int)blockIdx.x + step < n_tiles) t2 = a.tiles[blockIdx.x + step];
    int i = 0;
    for (int t = blockIdx.x; t < n_tiles; t += step, ++i) {
      const int buf = i & 1;
      const TcRow e = e1;
      EpiAdd nxt;
      epi_fetch(a, e, 0, nxt);
      if (t + step < n_tiles) e1 = epi_row(a, t2, row);
      if (t + 2 * step < n_tiles) t2 = a.tiles[t + 2 * step];
      bool ok = !*abort_v && mbar_wait(&acc_full[buf], (uint32_t)((i >> 1) & 1));
      ok = __all_sync(0xffffffffu, ok);   // tcgen05.ld below is warp-collective
      if (!ok) {
        if (lane == 0) {
          atomicCAS(a.err, 0, 16);
          *abort_v = 1;
        }
        break;
      }
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      epi_tile(a, tmem + (uint32_t)buf * a.tmem_cols + ((uint32_t)(quad * 32) << 16), e, nxt);
      // this warp's reads of the buffer are done: the MMA warp may overwrite it
      asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
      __syncwarp();
      if (lane == 0) mbar_arrive(&acc_empty[buf]);
    }
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (warp == 1) {
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(2u * a.tmem_cols)
                 : "memory");
  }
}

// Self-test of the bounded wait: waits on an mbarrier that expects two arrivals but receives
// one, so the phase never completes; the wait gives up after `limit` polls and the kernel
// reports MW_ETIMEOUT (5) in *code instead of hanging.
__global__ void bounded_wait_probe_kernel(long long limit, int32_t* code) {
  __shared__ __align__(8) uint64_t bar;
  if (threadIdx.x == 0) {
    mbar_init(&bar, 2);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(&bar)) : "memory");
    *code = mbar_wait(&bar, 0, limit) ? 0 : 5;
  }
}

inline int rpad(int R) { return (R + 7) / 8 * 8; }

}  // namespace

bool tc_plan_build(TcPlan& p, const mw::Subdomains& sd, const std::function<void*(size_t)>& alloc, int32_t* err,
                   cudaStream_t s) {
  p = TcPlan();
  const int ns = sd.n_sub;
  std::vector<TcTile> tiles;
  std::vector<int32_t> sub_kt(ns), gt_sub, gt_kt;
  std::vector<int64_t> sub_wtile(ns), sub_gtile(ns);
  int64_t wt = 0, gtile = 0;
  for (int q = 0; q < ns; ++q) {
    const int64_t n = sd.dof_ptr[q + 1] - sd.dof_ptr[q];
    const int64_t no = sd.own_ptr[q + 1] - sd.own_ptr[q];
    const int KT = (int)((n + kTileKd - 1) / kTileKd);
    const int MT = (int)((no + kTileM - 1) / kTileM);
    sub_kt[q] = KT;
    sub_wtile[q] = wt;
    sub_gtile[q] = gtile;
    for (int k = 0; k < KT; ++k) {
      gt_sub.push_back(q);
      gt_kt.push_back(k);
    }
    wt += (int64_t)MT * KT * 2;   // Wr and Wi tile per (m tile, k tile)
    gtile += KT;
  }
  p.n_sub = ns;
  // Output tiles by subdomain; longest first (most k tiles) when they make at most two waves of two
  // blocks per SM, so that the launch does not end on its longest: 32 subdomains of 2734 unknowns (350 tiles)
  // 103 -> 91 us per apply.  Longer launches keep the order: sorted they lost up to 5 % at 64 columns.
  std::vector<int32_t> order(ns);
  int64_t n_mtiles = 0;
  for (int q = 0; q < ns; ++q) {
    order[q] = q;
    n_mtiles += (sd.own_ptr[q + 1] - sd.own_ptr[q] + kTileM - 1) / kTileM;
  }
  if (n_mtiles <= 2 * 2 * 152)
    std::stable_sort(order.begin(), order.end(), [&](int a, int b) { return sub_kt[a] > sub_kt[b]; });
  for (int q : order) {
    const int64_t nown = sd.own_ptr[q + 1] - sd.own_ptr[q];
    for (int64_t r = 0; r < nown; r += kTileM)
      tiles.push_back({sub_wtile[q] + r / kTileM * sub_kt[q] * 2, sub_gtile[q], sd.own_ptr[q] + r, sub_kt[q],
                       (int32_t)std::min<int64_t>(kTileM, nown - r)});
  }
  p.n_mtiles = (int64_t)tiles.size();
  p.n_ktiles_total = gtile;
  p.w_tiles = wt;
  auto up = [&](const void* h, size_t bytes) {
    void* d = alloc(bytes);
    cudaMemcpyAsync(d, h, bytes, cudaMemcpyHostToDevice, s);
    return d;
  };
  if (tiles.empty()) tiles.resize(1);
  p.tiles = (TcTile*)up(tiles.data(), sizeof(TcTile) * tiles.size());
  p.sub_wtile = (int64_t*)up(sub_wtile.data(), sizeof(int64_t) * ns);
  p.sub_kt = (int32_t*)up(sub_kt.data(), sizeof(int32_t) * ns);
  p.gt_sub = (int32_t*)up(gt_sub.data(), sizeof(int32_t) * std::max<size_t>(gt_sub.size(), 1));
  p.gt_kt = (int32_t*)up(gt_kt.data(), sizeof(int32_t) * std::max<size_t>(gt_kt.size(), 1));
  p.err = err;
  cudaStreamSynchronize(s);  // host vectors go out of scope, and ring_open reads the records without waiting
  p.built = true;
  return true;
}

void tc_plan_free(TcPlan& p, const std::function<void(void*)>& dfree) {
  for (void* q : {(void*)p.tiles, (void*)p.sub_wtile, (void*)p.sub_kt,
                  (void*)p.gt_sub, (void*)p.gt_kt})
    if (q) dfree(q);
  p = TcPlan();
}

void bounded_wait_probe(long long limit, int32_t* code, cudaStream_t s) {
  note_launch(1);
  bounded_wait_probe_kernel<<<1, 32, 0, s>>>(limit, code);
}

size_t tc_w_bytes(const TcPlan& p) { return (size_t)std::max<int64_t>(p.w_tiles, 1) * kATileBytes; }

size_t tc_scratch_bytes(const TcPlan& p, int R) {
  return (size_t)std::max<int64_t>(p.n_ktiles_total, 1) * 2 * rpad(R) * 128;
}

void tc_extract(const TcPlan& p, const InvBatch& bt, const OrasTopo& tp, int ws_prec, const void* ws, void* W,
                cudaStream_t s) {
  note_launch(1);
  // grid: k tiles x m tiles of the largest subdomain in the batch x batch
  const int ktmax = (bt.np_max + kTileKd - 1) / kTileKd;
  const int mtmax = (bt.np_max + kTileM - 1) / kTileM;
  dim3 grid(ktmax, mtmax, bt.count);
  if (ws_prec == 0)
    pack_w_kernel<double2><<<grid, 256, 0, s>>>(bt, tp.own_ptr, tp.own_local, (const double2*)ws, p.sub_wtile,
                                                 p.sub_kt, (uint8_t*)W);
  else
    pack_w_kernel<float2><<<grid, 256, 0, s>>>(bt, tp.own_ptr, tp.own_local, (const float2*)ws, p.sub_wtile, p.sub_kt,
                                                (uint8_t*)W);
}

void tc_pack_stacked(const TcPlan& p, const MfTask* tasks, const int32_t* first, const int32_t* second,
                     const int64_t* own_ptr, const int32_t* own_local, int n, int ktmax, int mtmax, const float2* src,
                     void* W, cudaStream_t s) {
  for (int q0 = 0; q0 < n; q0 += 65535) {
    const int cnt = std::min(65535, n - q0);
    note_launch(1);
    dim3 grid((unsigned)std::max(ktmax, 1), (unsigned)std::max(mtmax, 1), (unsigned)cnt);
    pack_w_stacked_kernel<<<grid, 256, 0, s>>>(tasks, first, second, own_ptr, own_local, q0, p.sub_wtile, p.sub_kt,
                                               src, (uint8_t*)W);
  }
}

int tc_stages(int N);
size_t tc_smem_bytes(int N, int stages);

int tc_stages(int N) {
  // 110 KB of stages per CTA: two CTAs share the 228 KB of an SM (1 KB each for alignment and 1 KB reserved),
  // with three stages up to 16 columns (100 KB gave two: 39.7 against 36.4 us per apply of 27 subdomains, 16 columns)
  const int stage = 2 * kATileBytes + N * 128;
  int st = (110 * 1024) / stage;
  return st > 6 ? 6 : (st < 2 ? 2 : st);
}

// Most dynamic shared memory of an MMA block: 1 KB of the 227 KB is left for its static shared memory.
constexpr size_t kTcMaxSmem = (size_t)226 * 1024;

size_t tc_smem_bytes(int N, int stages) { return (size_t)stages * (2 * kATileBytes + N * 128) + 1024; }


int tc_max_stages(int R) {
  // the kernel holds 8 stage barriers
  const int N = 2 * rpad(R);
  int st = tc_min_stages;
  while (st < 8 && tc_smem_bytes(N, st + 1) <= kTcMaxSmem) ++st;
  return st;
}

// The MMA kernel over the plan's tiles, its operand tiles already in a.Bt.
static void tc_mma(const TcPlan& p, TcArgs a, int R, int stages, bool persistent, cudaStream_t s) {
  const int N = 2 * rpad(R);
  // one block per SM at most: the whole shared memory for its ring (117 tiles, 16 columns: 34.2 -> 33.3 us per apply)
  if (stages <= 0) stages = p.n_mtiles <= 152 ? tc_max_stages(R) : tc_stages(N);
  if (stages < tc_min_stages) stages = tc_min_stages;
  if (stages > tc_max_stages(R)) stages = tc_max_stages(R);
  note_launch(1);
  a.tiles = p.tiles;
  a.R = R;
  a.N = N;
  a.stages = stages;
  uint32_t cols = 32;
  while ((int)cols < 2 * N) cols <<= 1;   // two accumulators of N columns
  a.tmem_cols = cols;
  a.err = p.err;
  if (persistent && 2 * cols <= 512) {
    // two accumulator buffers per CTA; two CTAs per SM while both fit the 512 columns
    const int per_sm = 4 * cols <= 512 ? 2 : 1;
    size_t smem = tc_smem_bytes(N, stages);
    if (per_sm == 1 && smem < (size_t)120 * 1024) smem = (size_t)120 * 1024;
    static SmemLimit limit;
    limit.raise(oras_tc_persistent_kernel, kTcMaxSmem);
    const int grid = (int)std::min<int64_t>(p.n_mtiles, (int64_t)per_sm * 152);
    launch_chained(oras_tc_persistent_kernel, (unsigned)std::max(grid, 1), kThreadsTc, smem, s, a,
        (int)p.n_mtiles);
    return;
  }
  // two CTAs of an SM must fit their tensor memory (512 columns per SM): above 256 columns the
  // shared-memory request keeps one CTA per SM
  size_t smem = tc_smem_bytes(N, stages);
  if (cols > 256 && smem < (size_t)120 * 1024) smem = (size_t)120 * 1024;
  static SmemLimit limit;
  limit.raise(oras_tc_kernel, kTcMaxSmem);
  launch_chained(oras_tc_kernel, (unsigned)p.n_mtiles, kThreadsTc, smem, s, a);
}

void oras_apply_tc(const TcPlan& p, const OrasTopo& tp, const void* W, const float2* r, float2* z, int R,
                   void* scratch, cudaStream_t s, int stages, const double* in_scale, bool z_bf16,
                   const int32_t* go) {
  const int Rp = rpad(R);
  note_launch(1);
  const size_t gsm = (size_t)2 * Rp * 128;   // at most 32 KB
  const int64_t gblocks = std::min<int64_t>(p.n_ktiles_total, 152 * 8);    // one resident wave
  // the MMA kernel comes in while the gather runs where it has at most two waves of blocks: 27 subdomains, 16 columns
  // 33.9 -> 32.3 us; 731 tiles lost 0.4 % of a gradient evaluation
  const bool early = p.n_mtiles <= 2 * 2 * 152;
  launch_chained(gather_b_kernel, (unsigned)std::max<int64_t>(gblocks, 1), 128, gsm, s, p.gt_sub, p.gt_kt,
      tp.dof_ptr, tp.dofs, r, R, Rp, (uint8_t*)scratch, in_scale, p.n_ktiles_total, go, early);
  TcArgs a{};
  a.own_glob = tp.own_glob;
  a.z_bf16 = z_bf16 ? 1 : 0;
  a.go = go;
  a.early = early;
  a.vec = R % (z_bf16 ? 4 : 2) == 0 && ((uintptr_t)z & 15) == 0;
  a.W = (const uint8_t*)W;
  a.Bt = (const uint8_t*)scratch;
  a.z = z;
  tc_mma(p, a, R, stages, false, s);
}

void tc_sweep(const TcPlan& p, const TcRow* rows, const int32_t* src, int n_src, const void* W, const float2* in,
              float2* arena, float2* z, int R, void* scratch, cudaStream_t s, bool persistent) {
  const int Rp = rpad(R);
  note_launch(1);
  const unsigned blocks = (unsigned)p.n_ktiles_total, threads = (unsigned)std::min(8 * Rp, 256);
  const size_t gsm = (size_t)2 * Rp * 128;   // at most 32 KB
  if (n_src == 3)
    launch_chained(gather_rows_kernel<3>, blocks, threads, gsm, s, src, in, arena, R, Rp, (uint8_t*)scratch);
  else
    launch_chained(gather_rows_kernel<1>, blocks, threads, gsm, s, src, in, arena, R, Rp, (uint8_t*)scratch);
  TcArgs a{};
  a.rows = rows;
  a.vec = R % 2 == 0 && (((uintptr_t)arena | (uintptr_t)z) & 15) == 0;
  a.W = (const uint8_t*)W;
  a.Bt = (const uint8_t*)scratch;
  a.z = arena;
  a.z2 = z;
  tc_mma(p, a, R, 0, persistent, s);
}

// ---------------------------------------------------------------------------------------
// Fixed scratch for the preconditioner apply that allocates nothing.
//
// Some callers cannot allocate device memory when they apply the preconditioner: code that
// runs while another framework owns the whole device heap, code that forbids allocation after
// initialisation (latency-critical or embedded loops), or callers on paths where an allocation
// would synchronise the device.  For them the gathered operand of the tensor-core apply lives
// in this file-scope array instead of a context buffer.  Every GPU that loads the library holds
// it until the process exits.  All calls share it and it keeps the last call's contents; the
// gather kernel rewrites every byte a call reads (zero padding included), so nothing needs
// clearing, but calls that overlap on the GPU race on it.
// ---------------------------------------------------------------------------------------
static __device__ __align__(256) unsigned char g_noalloc_scratch[kNoAllocScratchBytes];

bool tc_noalloc_scratch(void** ptr, std::string& err) {
  // In host code the array's name is only a host-side handle; the device address is looked up
  // once per device, with that device current, and cached.
  static std::mutex mu;
  static void* addr[256] = {};
  int dev = -1;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess || dev < 0 || dev >= 256) {
    err = std::string("cudaGetDevice failed: ") + cudaGetErrorString(e);
    return false;
  }
  std::lock_guard<std::mutex> lock(mu);
  if (!addr[dev]) {
    void* p = nullptr;
    e = cudaGetSymbolAddress(&p, g_noalloc_scratch);
    if (e != cudaSuccess || !p) {
      err = std::string("cudaGetSymbolAddress of the fixed scratch failed: ") + cudaGetErrorString(e);
      return false;
    }
    addr[dev] = p;
  }
  *ptr = addr[dev];
  return true;
}

}  // namespace mwk

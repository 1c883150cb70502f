// BF16 tensor-core (tcgen05) form of the ORAS apply (K4): layout plan and launchers.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include <functional>
#include <string>

namespace mw {
struct Subdomains;
}

namespace mwk {
struct OrasTopo;
struct InvBatch;

// One 128-row output tile as the MMA kernels read it: everything a role needs in one 32-byte record.
struct alignas(16) TcTile {
  int64_t w;      // first W tile (Wr of k tile 0)
  int64_t g;      // first gathered-operand tile
  int64_t own;    // its first row in the owned-row lists
  int32_t kt;     // k tiles
  int32_t rows;   // rows that are owned, 1..128
};

// Pre-tiled BF16 layout of the owned-row inverses W_s (see k_oras_tc.cu).
struct TcPlan {
  bool built = false;
  int n_sub = 0;
  int64_t n_mtiles = 0;       // sum_s ceil(n_own_s / 128)
  int64_t n_ktiles_total = 0; // sum_s ceil(2 n_s / 64)
  int64_t w_tiles = 0;        // sum_s mtiles_s * ktiles_s (16 KB each)
  // device arrays
  TcTile* tiles = nullptr;       // [n_mtiles] output tiles in launch order
  int64_t* sub_wtile = nullptr;  // [n_sub] first W tile of s
  int32_t* sub_kt = nullptr;     // [n_sub] k tiles of s
  int32_t* gt_sub = nullptr;     // [n_ktiles_total] subdomain of each gathered-operand tile
  int32_t* gt_kt = nullptr;      // [n_ktiles_total] its k tile
  int32_t* err = nullptr;        // error word (mapped host memory): nonzero after a timed-out wait
};

// err: device address of the error word, kept by the caller.
bool tc_plan_build(TcPlan& p, const mw::Subdomains& sd, const std::function<void*(size_t)>& alloc, int32_t* err,
                   cudaStream_t s);
void tc_plan_free(TcPlan& p, const std::function<void(void*)>& dfree);
size_t tc_w_bytes(const TcPlan& p);
size_t tc_scratch_bytes(const TcPlan& p, int R);
void tc_extract(const TcPlan& p, const InvBatch& bt, const OrasTopo& tp, int ws_prec, const void* ws, void* W,
                cudaStream_t s);
struct MfTask;
// Packs the FP32 blocks of tasks (A = src + a_off, [m][k], row stride lda, times the task's
// sign) into the plan's BF16 tiles for n plan "subdomains" that each stack up to two products
// with the same B (same k): subdomain q is task first[q] over task second[q] (second[q] < 0: the
// first alone), and its output row i (own_ptr[q] <= i < own_ptr[q + 1]) is row own_local[i] of the
// stack; ktmax / mtmax: the largest tile counts.
void tc_pack_stacked(const TcPlan& p, const MfTask* tasks, const int32_t* first, const int32_t* second,
                     const int64_t* own_ptr, const int32_t* own_local, int n, int ktmax, int mtmax, const float2* src,
                     void* W, cudaStream_t s);
// Where an output row of a sweep goes: row out of the arena and row z of the result (-1: neither), after the
// arena rows add0 and add1 (-1: none) have been added.
struct alignas(16) TcRow {
  int32_t out, add0, add1, z;
};
// One launch of the sparse sweeps: the plan's products with operand rows from src, n_src (1 or 3) entries per
// row, summed in order (>= 0: that arena row, -1: nothing, else row -2 - src of in); 64 rows per k tile, in
// the order of the plan's k tiles.  in and z do not overlap.
// persistent: CTAs loop over the output tiles with one copy ring and double-buffered accumulators (for plans
// of many short tiles; up to 64 columns, else the one-tile-per-CTA kernel runs); the same bits either way.
void tc_sweep(const TcPlan& p, const TcRow* rows, const int32_t* src, int n_src, const void* W, const float2* in,
              float2* arena, float2* z, int R, void* scratch, cudaStream_t s, bool persistent);
// stages: shared-memory pipeline depth of the MMA kernel (0 = default; the result does not depend
// on it, only the speed).  in_scale (may be null): per-column factor of r (z = M^{-1}(r * in_scale)).
// z_bf16: z is written as complex BF16 pairs (real in the low half), 4 bytes per value, row stride R values.
// go (may be null): device word; zero when the kernels start: nothing is done.
void oras_apply_tc(const TcPlan& p, const OrasTopo& tp, const void* W, const float2* r, float2* z, int R,
                   void* scratch, cudaStream_t s, int stages = 0, const double* in_scale = nullptr,
                   bool z_bf16 = false, const int32_t* go = nullptr);
// Pipeline depths the MMA kernel accepts for R columns: [tc_min_stages, tc_max_stages(R)].
constexpr int tc_min_stages = 2;
int tc_max_stages(int R);

// Launches the bounded-wait self-test (see k_oras_tc.cu); *code (device) gets 0 or 5.
void bounded_wait_probe(long long limit, int32_t* code, cudaStream_t s);

// Size of the fixed scratch used by mw_apply_preconditioner_noalloc (16 MiB).
constexpr size_t kNoAllocScratchBytes = (size_t)16 << 20;
// Device address of the fixed scratch on the current device (looked up once per device).
bool tc_noalloc_scratch(void** ptr, std::string& err);

}  // namespace mwk

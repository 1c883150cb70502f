// Dense subdomain inverses of the ORAS setup (k_inverse.cu).
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include "k_oras.h"

namespace mwk {

// Unknowns per pivot block, and the multiple to which a matrix is padded.
constexpr int kInvBlock = 32, kInvPad = 64;

// A batch of subdomains whose matrices share one workspace (layout: see k_inverse.cu).
struct InvBatch {
  int count, steps, np_max;   // matrices, pivot blocks and padded order of the largest
  const int32_t* d_sub;       // [count] subdomain ids
  const int32_t* d_n;         // [count] unknowns n
  const int32_t* d_np;        // [count] n padded to a multiple of kInvPad
  const int64_t* d_off;       // [count] element offset of each matrix [np][np] in the workspace
  const int64_t* d_poff;      // [count] element offset of its panels [2][kInvBlock][np]
  const int32_t* d_nsw;       // [steps][count] owned unknowns before the step's pivot block
  const int32_t* d_prefix;    // [steps][count + 1] running tile counts of the step's update
  const int32_t* h_tiles;     // [steps] their totals (host)
};
// Tiles of the update of pivot block kb in a matrix of n unknowns (padded np), nsw owned ones before it.
int64_t inv_update_tiles(int n, int np, int nsw, int kb);

// zc (optional): coefficients of the outer-face classes (surf_tet = -1 - class); metal
// (optional, [E]): edges whose local rows and columns become those of the identity.  The workspace
// is zero on entry.  prec: 0 FP64, 1 FP32.
void oras_local_assemble(const InvBatch& bt, const OrasTopo& tp, const double* Bsurf, const double* KM,
                         const double* eps, double k0, double eps_bg_re, double eps_bg_im, const double2* zc,
                         const uint8_t* metal, int prec, void* ws, cudaStream_t s);
// dinv: count * kInvBlock^2 elements.
void oras_invert(const InvBatch& bt, const OrasTopo& tp, int prec, void* ws, void* dinv, int32_t* status,
                 cudaStream_t s);
void oras_extract(const InvBatch& bt, const OrasTopo& tp, int ws_prec, const void* ws, int w_prec,
                  const int64_t* w_off, void* W, cudaStream_t s);

}  // namespace mwk

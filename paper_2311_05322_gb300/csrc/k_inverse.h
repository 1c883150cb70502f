// Dense subdomain inverses of the ORAS setup (k_inverse.cu).
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include "k_oras.h"

namespace mwk {

// Pivot block sizes of the FP32 and FP64 factorisations.
constexpr int kInvBlock32 = 64, kInvBlock64 = 32;
int inv_block(int prec);

// A batch of subdomains whose matrices share one workspace (positions: see k_inverse.cu).
struct InvBatch {
  int count, steps, np_max;   // matrices, pivot blocks and order of the largest
  const int32_t* d_sub;       // [count] subdomain ids
  const int32_t* d_np;        // [count] padded order np (a multiple of the pivot block)
  const int32_t* d_mn;        // [count] padded count of the unknowns not owned
  const int64_t* d_off;       // [count] element offset of each matrix [np][np] in the workspace
  const int64_t* d_poff;      // [count] element offset of its panel [2][block][np]
  const int32_t* d_pos;       // position of every local unknown, at dof_ptr[s]
  const int32_t* d_prefix;    // [steps][count + 1] running tile counts of the step's update
  const int32_t* h_tiles;     // [steps] their totals (host)
};
// Tiles of the update of pivot block kb in a matrix of order np with mn unknowns not owned.
int64_t inv_update_tiles(int np, int mn, int kb);

// zc (optional): coefficients of the outer-face classes (surf_tet = -1 - class); metal
// (optional, [E]): edges whose local rows and columns become those of the identity.  The workspace
// is zero on entry.  prec: 0 FP64, 1 FP32.
void oras_local_assemble(const InvBatch& bt, const OrasTopo& tp, const double* Bsurf, const double* KM,
                         const double* eps, double k0, double eps_bg_re, double eps_bg_im, const double2* zc,
                         const uint8_t* metal, int prec, void* ws, cudaStream_t s);
// dinv: 2 * count * block * block elements.
void oras_invert(const InvBatch& bt, int prec, void* ws, void* dinv, int32_t* status, cudaStream_t s);
void oras_extract(const InvBatch& bt, const OrasTopo& tp, int ws_prec, const void* ws, int w_prec,
                  const int64_t* w_off, void* W, cudaStream_t s);

}  // namespace mwk

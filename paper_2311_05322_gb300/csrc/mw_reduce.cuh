// Sums over a block's rows, per column, of the kernels that map threads to (row, column).
#pragma once

namespace mwk {

// The block (256 threads) holds in thread t, nrm[q] for column c0 + q cstep of one row, with c0 a function of
// t % tpr; the sums over the rows go to out[column] for columns below R.  Over the rows of each warp by
// shuffles, then over the 8 warps: a serial sum over the block's rows (64 of them at 3 columns) waited for 64
// FP64 adds in turn, 2 us.  red: 256 CPL doubles of shared memory.
template <int CPL>
__device__ __forceinline__ void store_column_norms(double (&nrm)[CPL], double* red, int tpr, int c0, int cstep, int R,
                                                   double* __restrict__ out) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
#pragma unroll
  for (int q = 0; q < CPL; ++q) {
    for (int off = tpr; off < 32; off <<= 1) nrm[q] += __shfl_xor_sync(0xffffffffu, nrm[q], off);
    if (lane < tpr) red[(warp * tpr + lane) * CPL + q] = nrm[q];
  }
  __syncthreads();
  if ((int)threadIdx.x < tpr)
#pragma unroll
    for (int q = 0; q < CPL; ++q) {
      const int c = c0 + q * cstep;
      if (c >= R) continue;
      double s = 0.0;
#pragma unroll
      for (int w = 0; w < 8; ++w) s += red[(w * tpr + (int)threadIdx.x) * CPL + q];
      out[c] = s;
    }
}

}  // namespace mwk

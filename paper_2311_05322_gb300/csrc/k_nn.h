// Launchers of the learned-initialiser kernels (k_nn.cu).
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

namespace mwk {
// Dense layers with BF16 weights W [N][K], FP32 elsewhere.  ws (ws_floats floats): partial sums of a
// split K, used when the tile grid alone would leave SMs idle; the split sums in a fixed order.
// h [B][N] = relu(x [B][K] W^T + bias)
void nn_dense_fwd(const float* x, const void* W, const float* bias, float* h, int B, int N, int K, float* ws,
                  size_t ws_floats, cudaStream_t s);
// dx [B][K] = dz [B][N] W where h [B][K] > 0, else 0 (h: the ReLU output that entered the layer)
void nn_dense_bwd_data(const float* dz, const void* W, const float* h, float* dx, int B, int N, int K, float* ws,
                       size_t ws_floats, cudaStream_t s);
// dW [N][K] = dz^T x
void nn_dense_bwd_w(const float* dz, const float* x, float* dW, int B, int N, int K, float* ws, size_t ws_floats,
                    cudaStream_t s);
void nn_colsum(const float* dz, int B, int N, float* db, cudaStream_t s);
// The decoder's transposed convolutions, layer 0: 16 -> 16 at 4^3, 1: 16 -> 8 at 8^3, 2: 8 -> 2 at
// 16^3 (input positions).  Forward: y, after the ReLU for layers 0 and 1.
void nn_convT_fwd(int layer, const float* x, const float* w, const float* b, float* y, int B, cudaStream_t s);
// Backward from dy: weight and bias gradients, and dx masked by the ReLU that made x (0 where x is
// not positive).  part: B * 16 floats of per-(channel, sample) partial sums for the bias
// gradient; wpart: kConvChunks * 16 * 16 * 64 floats of partial weight-gradient sums.
constexpr int kConvChunks = 64;
void nn_convT_bwd(int layer, const float* x, const float* w, const float* dy, float* dx, float* dw, float* db, int B,
                  float* part, float* wpart, cudaStream_t s);
void nn_mse(const float* y, const float* t, int64_t n, float* dy, double* part, double* loss, cudaStream_t s);
void nn_adam(float* th, const float* g, float* m, float* v, int64_t n, float lr, float b1, float b2, float eps, int step,
             cudaStream_t s);
void nn_to_bf16(const float* a, void* b, int64_t n, cudaStream_t s);
void nn_gather_rows(const float* src, const int32_t* idx, int n, int64_t width, float* dst, cudaStream_t s);
void nn_grid_to_tets(const float* grid, int G, const double* box, const double* xyz, const int32_t* tets, int64_t T,
                     double* out, cudaStream_t s);
}  // namespace mwk

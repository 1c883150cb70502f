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
// The decoder's transposed convolutions, layer 0: 16 -> 16 at 4^3, 1: 16 -> 8 at 8^3, 2: 8 -> 2 at
// 16^3 (input positions).  Forward: y, after the ReLU for layers 0 and 1.
void nn_convT_fwd(int layer, const float* x, const float* w, const float* b, float* y, int B, cudaStream_t s);
// Backward from dy: dx masked by the ReLU that made x (0 where x is not positive), and the partial
// sums of the weight and bias gradients that nn_final_sums completes.  bpart: 26 B floats; wpart:
// kConvChunks * 400 * 64 floats (all three layers).
constexpr int kConvChunks = 64;
void nn_convT_bwd(int layer, const float* x, const float* w, const float* dy, float* dx, int B, float* bpart,
                  float* wpart, cudaStream_t s);
// The second-pass sums of a backward pass: weight and bias gradients of the three layers, and the
// dense layers' bias gradients db1, db2 = column sums of dz1, dz2 [B][N].
void nn_final_sums(int B, const float* bpart, const float* wpart, float* const dw[3], float* const db[3],
                   const float* dz1, const float* dz2, int N, float* db1, float* db2, cudaStream_t s);
// y, dy [B][width] against rows idx[b] of t (rows b without idx); width a multiple of 4096; part: B *
// width / 4096 doubles; *loss = mean of (y - t)^2.
void nn_mse(const float* y, const float* t, const int32_t* idx, int B, int64_t width, float* dy, double* part,
            double* loss, cudaStream_t s);
// Adam on n parameters; the entries [0, n1) and [o2, o2 + n2) (multiples of 4) also go to the BF16 copies
// w1 and w2.
void nn_adam(float* th, const float* g, float* m, float* v, void* w1, void* w2, int64_t n, int64_t n1, int64_t o2,
             int64_t n2, float lr, float b1, float b2, float eps, int step, cudaStream_t s);
void nn_to_bf16(const float* a, void* b, int64_t n, cudaStream_t s);
void nn_gather_rows(const float* src, const int32_t* idx, int n, int64_t width, float* dst, cudaStream_t s);
void nn_grid_to_tets(const float* grid, int G, const double* box, const double* xyz, const int32_t* tets, int64_t T,
                     double* out, cudaStream_t s);
}  // namespace mwk

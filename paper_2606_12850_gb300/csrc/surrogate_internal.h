// Internal declarations of the surrogate network's CUDA kernels (surrogate_kernels.cu),
// used by the model runtime (surrogate_capi.cpp). Activations are float32 [batch][C][L]
// (or [batch][features]); weights are read as bfloat16; every reduction runs in a fixed
// order, so results are bitwise reproducible.
#pragma once

#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <cstddef>

namespace sgk {

using bf16 = __nv_bfloat16;

constexpr int kSms = 152;  // GB300

// How the products run. kind 0: warp-level mma.sync, 128/256 x 64 tiles. kind 1: tcgen05 with
// the accumulator in tensor memory, 128 x 128 tiles. Both round the operands to bfloat16
// (nearest even) and accumulate in float32. err: a device word that a kind-1 product sets to 1
// when one of its bounded waits for the tensor cores runs out (required for kind 1).
// pack: device scratch of pack_bytes for the convolutions' packed weights (kind 1; at least
// conv_pack_bytes of every layer).
struct Products {
  int kind = 1;
  int* err = nullptr;
  int stall_test = 0;  // 1: every kind-1 product waits for a phase nothing completes (tests the limit)
  bf16* pack = nullptr;
  size_t pack_bytes = 0;
  float* red = nullptr;   // scratch of red_floats for the bias gradients' per-slice sums
  size_t red_floats = 0;
  size_t ws_floats = 0;   // capacity of the split-K workspace a call receives (splits are clamped to it)
};
// Bytes of the packed weights of a convolution with Ci input and Co output channels.
size_t conv_pack_bytes(int Ci, int Co);

// Split-K workspace need (floats) of the weight-gradient products for an M x N result.
size_t splitk_floats(int M, int N, int K);

// Y = act(X W^T + b): X [B][K], W [N][K] (bf16), pre/out [B][N]; out may alias nothing.
int linear_forward(int B, int K, int N, const float* X, const bf16* W, const float* bias, float* pre, float* out,
                   bool gelu, const Products& pr, cudaStream_t s);
// dX [B][K] = dZ [B][N] W [N][K]; split over N through ws (splitk_floats(B, K, N)) when given
int linear_backward_data(int B, int K, int N, const float* dZ, const bf16* W, float* dX, float* ws,
                         const Products& pr, cudaStream_t s);
// dW [N][K] = dZ^T X; db [N] = column sums of dZ
int linear_backward_weight(int B, int K, int N, const float* dZ, const float* X, float* dW, float* db, float* ws,
                           const Products& pr, cudaStream_t s);

// Width-3 'same' convolution of the input upsampled by `up` along time:
// pre[b][o][t] = bias[o] + sum_{c,d} W[o][c][d] X[b][c][(t + d - 1) / up] (zero outside),
// t < L = Lin * up; out = gelu(pre) when out != nullptr. Kind 1 runs its own tcgen05 kernel
// (the input window staged once for the three taps), kind 0 the generic product.
int conv_forward(int B, int Ci, int Co, int Lin, int up, const float* X, const bf16* W, const float* bias,
                 float* pre, float* out, const Products& pr, cudaStream_t s);
// dX [B][Ci][Lin] from dZ [B][Co][L] (the upsampling adjoint sums the repeated samples)
int conv_backward_data(int B, int Ci, int Co, int Lin, int up, const float* dZ, const bf16* W, float* dX,
                       const Products& pr, cudaStream_t s);
// dW [Co][Ci][3] and db [Co]
int conv_backward_weight(int B, int Ci, int Co, int Lin, int up, const float* dZ, const float* X, float* dW,
                         float* db, float* ws, const Products& pr, cudaStream_t s);

// dz[i] *= gelu'(pre[i])
int gelu_backward(size_t n, const float* pre, float* dz, cudaStream_t s);
// dy = 2 (y - t) / n; partials[kLossBlocks] = per-block sums of (y - t)^2 in float64
constexpr int kLossBlocks = 608;
int mse_grad(size_t n, const float* y, const float* t, float* dy, double* partials, cudaStream_t s);
// Adam on n master parameters, then the bf16 mirror
int adam_update(size_t n, float* p, const float* g, float* m, float* v, bf16* pb, float lr, float beta1, float beta2,
                float eps, float inv_c1, float inv_c2, cudaStream_t s);
int to_bf16(size_t n, const float* p, bf16* pb, cudaStream_t s);
// y [B][C][L] = sum_k x[b][in_dim - K + k] D[b][k*C + c][t], and its adjoint in D
int contract_forward(int B, int K, int C, int L, int in_dim, const float* x, const float* D, float* y, cudaStream_t s);
int contract_backward(int B, int K, int C, int L, int in_dim, const float* x, const float* dy, float* dD,
                      cudaStream_t s);

// ---- packed passes (surrogate_packed.cu): bfloat16 activations in the tensor cores' layout ----
// rows of a packed time axis of L samples (one zero row before, zeros after)
int packed_rows(int L);
bool packed_dense_ok(int K, int N);
bool packed_conv_ok(int Ci, int N, int up);
size_t packed_dense_elems(int K, int N);  // packed weights of a dense layer
// W [N][K] -> packed; l0 > 0: the layer feeds a convolution of N / l0 channels
int pack_dense(int K, int N, int l0, const bf16* W, bf16* Wp, cudaStream_t s);
// W [Co][Ci][3] -> packed blocks of N rows; outC > 0: contracted copies of 32 channels a block
int pack_conv(int Ci, int N, int blocks, int outC, const bf16* W, bf16* Wp, cudaStream_t s);
// out = gelu(x W^T + b), from x [B][K] (or, x null, packed [K/8][Bp][8]) to packed [N/8][Bp][8]
// (or, l0 > 0, [B][N/l0/8][packed_rows(l0)][8]); pre and act (or null) [B][N]
int packed_dense(int B, int Bp, int K, int N, const float* x, const bf16* in, const bf16* Wp, const float* bias,
                 bf16* out, float* pre, float* act, int l0, const Products& pr, cudaStream_t s);
// hidden convolution, packed to packed; pre (or null) [B][N][up Lin]
int packed_conv(int B, int Ci, int N, int Lin, int up, const bf16* in, const bf16* Wp, const float* bias, bf16* out,
                float* pre, const Products& pr, cudaStream_t s);
// the last convolution (K outC channels, no upsampling) and its contraction with x: y [B][outC][Lin]
int packed_conv_contract(int B, int Ci, int K, int outC, int Lin, int in_dim, const bf16* in, const bf16* Wp,
                         const float* bias, const float* x, float* y, const Products& pr, cudaStream_t s);
// The same in training: the sum of squared errors against target [B][outC][Lin] (loss, a value
// per block of packed_loss_blocks), the packed gradient dD of the K outC channels and their bias
// gradients db; row_sums: scratch of B * 4 ceil(Lin / 128) * outC floats
int packed_loss(int B, int Ci, int K, int outC, int Lin, int in_dim, const bf16* in, const bf16* Wp, const float* bias,
                const float* x, const float* target, bf16* dD, float* row_sums, float* db, double* loss,
                const Products& pr, cudaStream_t s);
int packed_loss_blocks(int B, int outC, int Lin);
// values the loss buffer holds: what mse_grad and packed_loss leave there for any batch up to B
// (past kSms column blocks packed_loss has a CTA per 32 channels, more than kLossBlocks of them
// from 19488 channels on)
int loss_values(int B, int outC, int Lin);
bool packed_backward_ok(int Ci, int Co, int up);
size_t packed_grad_elems(int Co, int Lin, int up);  // packed gradient of one sample, [Co/8][up][rows][8]
int pack_conv_t(int Ci, int Co, const bf16* W, bf16* Wt, cudaStream_t s);
// dW [Co][Ci][3] from the packed gradient dZ of the output and the packed input X
int packed_conv_wgrad(int B, int Ci, int Co, int Lin, int up, const bf16* dZ, const bf16* X, float* dW, float* ws,
                      const Products& pr, cudaStream_t s);
// The gradient at the layer below: dz = dX gelu'(pre), packed (out, of a layer that upsamples by
// out_up) or float32 [B][Ci][Lin] (out_f32), and its bias gradients db [Ci] (sums: scratch of kSms
// Ci floats; both null to leave them out)
int packed_conv_dgrad(int B, int Ci, int Co, int Lin, int up, const bf16* dZ, const bf16* Wt, const float* pre,
                      bf16* out, int out_up, float* out_f32, float* sums, float* db, const Products& pr,
                      cudaStream_t s);

}  // namespace sgk

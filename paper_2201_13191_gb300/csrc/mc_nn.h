// Launch wrappers of the denoiser's element-wise kernels (k_nn.cu).
#pragma once
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stddef.h>
#include <stdint.h>

namespace mcx {
namespace nn {

cudaError_t image_mean(const float* img, int n, int hw, float* scale, cudaStream_t s);
cudaError_t pack_input(const float* img, const float* scale, int n, int hw, __nv_bfloat16* x, cudaStream_t s);
cudaError_t unpack_output(const float* img, const float* scale, const float* net, int n, int hw, float* out,
                          cudaStream_t s);
// Loss of a batch; the output gradient in BF16 [n][hw][16] and its bias gradient db[0] (added to).
cudaError_t mse(const float* img, const float* tgt, const float* scale, const float* net, int n, int hw,
                __nv_bfloat16* gb, float* db, double* loss, cudaStream_t s);
// Gradient at a layer's output y ([n][h][w][c], c a power of two in 16 .. 256) through its ReLU, in BF16, with the bias
// gradient added to db.  PLAIN: g [n][h][w][c]; UP: y was up-sampled by 2, g [n][2h][2w][c]; POOL: y was also pooled,
// gp [n][h/2][w/2][c].
enum MaskMode { MASK_PLAIN = 0, MASK_UP = 1, MASK_POOL = 2 };
cudaError_t mask(MaskMode mode, const float* g, const float* gp, const __nv_bfloat16* y, int n, int h, int w, int c,
                 __nv_bfloat16* gb, float* db, cudaStream_t s);
cudaError_t pool_fwd(const __nv_bfloat16* x, int n, int h, int w, int c, __nv_bfloat16* y, cudaStream_t s);
// y [n][2h][2w][c + cs] = (x [n][h][w][c] up-sampled by 2, skip [n][2h][2w][cs])
cudaError_t up_concat(const __nv_bfloat16* x, const __nv_bfloat16* skip, int n, int h, int w, int c, int cs,
                      __nv_bfloat16* y, cudaStream_t s);
// Every layer's parameters in one array: layer l at [begin[l], begin[l + 1]), weights [cout][9][cin] then biases; wf and
// wa its operand copies.
struct LayerTable {
  int layers;
  uint32_t begin[17];
  int cin[16], cout[16];
  __nv_bfloat16 *wf[16], *wa[16];
};
cudaError_t adam(float* w, const float* g, float* m, float* v, const LayerTable& t, float lr, int step, cudaStream_t s);
// Tensor-core operand order of the convolution weights (forward wf and adjoint
// wa, either nullable): wf[ci/8][tap][co][ci%8], wa[co/8][8-tap][ci][co%8].
cudaError_t pack_weights(const float* w, int cout, int cin, __nv_bfloat16* wf, __nv_bfloat16* wa, cudaStream_t s);
cudaError_t pack_weights_bf16(const __nv_bfloat16* w, int cout, int cin, __nv_bfloat16* wf, cudaStream_t s);

}  // namespace nn
}  // namespace mcx

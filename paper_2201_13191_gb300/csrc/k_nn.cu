// Element-wise, pooling, resampling, loss and optimiser kernels of the learned
// scatter denoiser (NHWC tensors; activations BF16, gradients FP32).
#include <cuda_bf16.h>
#include <stdint.h>

#include "mc_nn.h"

namespace mcx {
namespace nn {
namespace {

__device__ __forceinline__ size_t gtid() { return (size_t)blockIdx.x * blockDim.x + threadIdx.x; }
__device__ __forceinline__ size_t gstride() { return (size_t)gridDim.x * blockDim.x; }
__device__ __forceinline__ __nv_bfloat16 to_bf(float v) { return __float2bfloat16_rn(v); }
__device__ __forceinline__ __nv_bfloat16 to_bf(__nv_bfloat16 v) { return v; }

int blocks_for(size_t n) {
  const size_t b = (n + 255) / 256;
  return (int)(b < 152 * 16 ? (b > 0 ? b : 1) : 152 * 16);
}

// Per-image scale: s[i] = mean of the image (floored at tiny > 0).  A thread
// adds its pixels one by one, but loads kMeanLoads of them at a time: the block
// is bound by the latency of its loads (256^2 image: 66 -> 9 us).
constexpr int kMeanLoads = 32;
__global__ void __launch_bounds__(256) k_image_mean(const float* __restrict__ img, int hw, float* __restrict__ s) {
  __shared__ float red[256];
  const float* im = img + (size_t)blockIdx.x * hw;
  float acc = 0.f;
  int i = threadIdx.x;
  for (; i + (kMeanLoads - 1) * 256 < hw; i += kMeanLoads * 256) {
    float v[kMeanLoads];
#pragma unroll
    for (int k = 0; k < kMeanLoads; ++k) v[k] = __ldg(im + i + k * 256);
#pragma unroll
    for (int k = 0; k < kMeanLoads; ++k) acc += v[k];
  }
  for (; i < hw; i += 256) acc += im[i];
  red[threadIdx.x] = acc;
  __syncthreads();
  for (int o = blockDim.x / 2; o > 0; o >>= 1) {
    if (threadIdx.x < o) red[threadIdx.x] += red[threadIdx.x + o];
    __syncthreads();
  }
  if (threadIdx.x == 0) s[blockIdx.x] = fmaxf(red[0] / (float)hw, 1e-30f);
}

// x[n][y][x][0] = img / s, other 15 channels 0.
__global__ void k_pack_input(const float* __restrict__ img, const float* __restrict__ s, int n, int hw,
                             __nv_bfloat16* __restrict__ x) {
  for (size_t i = gtid(); i < (size_t)n * hw; i += gstride()) {
    const int b = (int)(i / hw);
    __align__(16) __nv_bfloat16 v[16];
    v[0] = __float2bfloat16_rn(img[i] / s[b]);
#pragma unroll
    for (int c = 1; c < 16; ++c) v[c] = __float2bfloat16_rn(0.f);
    uint4* dst = reinterpret_cast<uint4*>(x + i * 16);
    dst[0] = reinterpret_cast<uint4*>(v)[0];
    dst[1] = reinterpret_cast<uint4*>(v)[1];
  }
}

// out = s * (img / s + net[...][0]) = img + s * net[...][0]   (residual output)
__global__ void k_unpack_output(const float* __restrict__ img, const float* __restrict__ s,
                                const float* __restrict__ net, int n, int hw, float* __restrict__ out) {
  for (size_t i = gtid(); i < (size_t)n * hw; i += gstride()) {
    const int b = (int)(i / hw);
    out[i] = img[i] + s[b] * net[i * 16];
  }
}

// Eight BF16 channels (16 bytes) as floats and back.
struct Eight {
  float v[8];
};
__device__ __forceinline__ Eight unpack8(uint4 q) {
  Eight e;
  const uint32_t w[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    e.v[2 * k] = __uint_as_float(w[k] << 16);
    e.v[2 * k + 1] = __uint_as_float(w[k] & 0xFFFF0000u);
  }
  return e;
}
__device__ __forceinline__ uint4 pack8(const float (&v)[8]) {
  __nv_bfloat162 b[4];
#pragma unroll
  for (int k = 0; k < 4; ++k) b[k] = __floats2bfloat162_rn(v[2 * k], v[2 * k + 1]);
  return *reinterpret_cast<uint4*>(b);
}
__device__ __forceinline__ void load8(const float* p, float (&v)[8]) {
  const float4 a = __ldg(reinterpret_cast<const float4*>(p)), b = __ldg(reinterpret_cast<const float4*>(p) + 1);
  v[0] = a.x; v[1] = a.y; v[2] = a.z; v[3] = a.w;
  v[4] = b.x; v[5] = b.y; v[6] = b.z; v[7] = b.w;
}

// Loss = mean over pixels of (x/s + net0 - y/s)^2; the gradient of the 16 output
// channels (channel 0 alone is used) goes out in BF16, as the convolutions'
// backward passes take it, and its sum into the bias gradient db[0].
__global__ void __launch_bounds__(256) k_mse(const float* __restrict__ img, const float* __restrict__ tgt,
                                             const float* __restrict__ s, const float* __restrict__ net, int n, int hw,
                                             uint4* __restrict__ gb, float* __restrict__ db, double* __restrict__ loss) {
  __shared__ double red[256];
  __shared__ float red_b[256];
  const float inv = 1.f / (float)((size_t)n * hw);
  double acc = 0.0;
  float bias = 0.f;
  for (size_t i = gtid(); i < (size_t)n * hw; i += gstride()) {
    const int b = (int)(i / hw);
    const float d = img[i] / s[b] + net[i * 16] - tgt[i] / s[b];
    acc += (double)d * d;
    const float v[8] = {2.f * d * inv, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
    const uint4 q = pack8(v);
    gb[2 * i] = q;
    gb[2 * i + 1] = make_uint4(0u, 0u, 0u, 0u);
    bias += __uint_as_float(q.x << 16);
  }
  red[threadIdx.x] = acc;
  red_b[threadIdx.x] = bias;
  __syncthreads();
  for (int o = blockDim.x / 2; o > 0; o >>= 1) {
    if (threadIdx.x < o) {
      red[threadIdx.x] += red[threadIdx.x + o];
      red_b[threadIdx.x] += red_b[threadIdx.x + o];
    }
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    atomicAdd(loss, red[0] * inv);
    atomicAdd(db, red_b[0]);
  }
}

// Gradient at a convolution's output, as its backward passes take it: gb =
// bf16(g [y > 0]) (the ReLU whose output is y) and db[c] += sum over pixels of gb.
//   MODE 0: g is the FP32 gradient [n][h][w][c] itself;
//   MODE 1: y was up-sampled by 2 (nearest): g [n][2h][2w][c] is summed 2 x 2;
//   MODE 2: y also went through 2 x 2 max pooling: the pooled gradient gp
//           [n][h/2][w/2][c] is added at the first maximum of each window.
// Eight channels per thread, so every access is 16 bytes or more, and nothing is
// stored in between (separate kernels with one channel per thread took 5.8 ms of
// a 19 ms pair of training steps at 16 x 256^2, of which this takes 1).  A thread
// keeps its channels from pixel to pixel (the stride is whole pixels) and their
// sums in registers.
constexpr int kMaskThreads = 256;
template <int MODE>
__global__ void __launch_bounds__(kMaskThreads) k_mask(const float* __restrict__ g, const float* __restrict__ gp,
                                                       const uint4* __restrict__ y, size_t npix, int h, int w, int c,
                                                       uint4* __restrict__ gb, float* __restrict__ db) {
  __shared__ float red[kMaskThreads / 32][256];
  const int cgs = c / 8, cg = threadIdx.x % cgs, lane = threadIdx.x & 31;
  // pixels of 2 x 2 windows in MODE 2, single pixels otherwise
  const int ow = MODE == 2 ? w / 2 : w, oh = MODE == 2 ? h / 2 : h;
  const size_t items = MODE == 2 ? npix / 4 : npix;
  const size_t step = (size_t)gridDim.x * (kMaskThreads / cgs);
  float sum[8] = {};
  auto put = [&](size_t pix, float (&v)[8], const Eight& yy) {
#pragma unroll
    for (int k = 0; k < 8; ++k) v[k] = yy.v[k] > 0.f ? v[k] : 0.f;
    const uint4 q = pack8(v);
    gb[pix * cgs + cg] = q;
    const Eight r = unpack8(q);
#pragma unroll
    for (int k = 0; k < 8; ++k) sum[k] += r.v[k];
  };
  for (size_t i = (size_t)blockIdx.x * (kMaskThreads / cgs) + threadIdx.x / cgs; i < items; i += step) {
    if (MODE == 0) {
      float v[8];
      load8(g + i * c + 8 * cg, v);
      put(i, v, unpack8(__ldg(y + i * cgs + cg)));
      continue;
    }
    const size_t t = i / ow;
    const int x = (int)(i - t * ow), yy = (int)(t % oh);
    const size_t b = t / oh;
    if (MODE == 1) {
      const float* p = g + (((b * (2 * h) + 2 * yy) * (2 * (size_t)w)) + 2 * x) * c + 8 * cg;
      float v[8], a[8];
      load8(p, v);
#pragma unroll
      for (int q = 1; q < 4; ++q) {
        load8(p + (q >> 1) * (2 * (size_t)w) * c + (q & 1) * c, a);
#pragma unroll
        for (int k = 0; k < 8; ++k) v[k] += a[k];
      }
      put(i, v, unpack8(__ldg(y + i * cgs + cg)));
    } else {
      float add[8];
      load8(gp + i * c + 8 * cg, add);
      Eight in[4];
      size_t pix[4];
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        pix[q] = (b * h + 2 * yy + (q >> 1)) * w + 2 * x + (q & 1);
        in[q] = unpack8(__ldg(y + pix[q] * cgs + cg));
      }
      int best[8];
#pragma unroll
      for (int k = 0; k < 8; ++k) {
        float m = in[0].v[k];
        best[k] = 0;
#pragma unroll
        for (int q = 1; q < 4; ++q)
          if (in[q].v[k] > m) {
            m = in[q].v[k];
            best[k] = q;
          }
      }
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        float v[8];
        load8(g + pix[q] * c + 8 * cg, v);
#pragma unroll
        for (int k = 0; k < 8; ++k) v[k] = best[k] == q ? v[k] + add[k] : v[k];
        put(pix[q], v, in[q]);
      }
    }
  }
  // lanes of the same channels, then the warps, then one add per channel
#pragma unroll
  for (int k = 0; k < 8; ++k)
    for (int o = 16; o >= cgs; o >>= 1) sum[k] += __shfl_xor_sync(0xffffffffu, sum[k], o);
  if (lane < cgs)
#pragma unroll
    for (int k = 0; k < 8; ++k) red[threadIdx.x >> 5][8 * cg + k] = sum[k];
  __syncthreads();
  for (int k = threadIdx.x; k < c; k += kMaskThreads) {
    float t = 0.f;
    for (int r = 0; r < kMaskThreads / 32; ++r) t += red[r][k];
    atomicAdd(db + k, t);
  }
}

// 2x2 max pooling (h, w even), one row of output pixels per block, eight channels per thread.
__global__ void __launch_bounds__(256) k_pool_fwd(const uint4* __restrict__ x, int w, int cgs, uint4* __restrict__ y) {
  const int per_row = (w / 2) * cgs;
  const uint4* r0 = x + (size_t)blockIdx.x * 2 * w * cgs;
  const uint4* r1 = r0 + (size_t)w * cgs;
  for (int i = threadIdx.x; i < per_row; i += blockDim.x) {
    const int xo = i / cgs, cg = i - xo * cgs, at = 2 * xo * cgs + cg;
    const Eight a = unpack8(__ldg(r0 + at)), b = unpack8(__ldg(r0 + at + cgs)), c = unpack8(__ldg(r1 + at)),
                d = unpack8(__ldg(r1 + at + cgs));
    float m[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) m[k] = fmaxf(fmaxf(fmaxf(a.v[k], b.v[k]), c.v[k]), d.v[k]);
    y[(size_t)blockIdx.x * per_row + i] = pack8(m);
  }
}

// A decoder level's input: y[..][0, c) = x up-sampled by 2 (nearest), y[..][c, c + cs) = the skip connection.  One row
// of output pixels per block, eight channels per thread (one channel per thread and separate kernels: 43% of a denoiser
// call; 1.73 -> 0.25 ms of a 40-image call at 256^2).
__global__ void __launch_bounds__(256) k_up_concat(const uint4* __restrict__ x, const uint4* __restrict__ skip, int h,
                                                   int w, int cgs, int sgs, uint4* __restrict__ y) {
  // output rows of 2 w pixels; h, w, x: the coarse level's
  const int tot = cgs + sgs, per_row = 2 * w * tot;
  const size_t b = blockIdx.x / (2 * h);
  const int Y = (int)(blockIdx.x - b * (2 * h));
  const uint4* xr = x + ((b * h + Y / 2) * w) * cgs;
  const uint4* sr = skip + (size_t)blockIdx.x * (2 * w) * sgs;
  uint4* yr = y + (size_t)blockIdx.x * per_row;
  for (int i = threadIdx.x; i < per_row; i += blockDim.x) {
    const int X = i / tot, k = i - X * tot;
    yr[i] = k < cgs ? __ldg(xr + (X / 2) * cgs + k) : __ldg(sr + X * sgs + (k - cgs));
  }
}

// Adam on every FP32 parameter of the network, in one launch (the parameters of
// all layers lie in one array, a layer's weights before its biases), with the
// BF16 operand copies of the weights (see k_pack_weights).
__global__ void __launch_bounds__(256) k_adam(float* __restrict__ w, const float* __restrict__ g, float* __restrict__ m,
                                              float* __restrict__ v, LayerTable t, float lr, float b1, float b2,
                                              float eps, float c1, float c2) {
  const uint32_t n = t.begin[t.layers];
  for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    const float gi = g[i];
    const float mi = b1 * m[i] + (1.f - b1) * gi;
    const float vi = b2 * v[i] + (1.f - b2) * gi * gi;
    m[i] = mi;
    v[i] = vi;
    const float wi = w[i] - lr * (mi / c1) / (sqrtf(vi / c2) + eps);
    w[i] = wi;
    int l = 0;
    while (i >= t.begin[l + 1]) ++l;
    const uint32_t k = i - t.begin[l], cin = (uint32_t)t.cin[l], cout = (uint32_t)t.cout[l];
    if (k >= cout * 9u * cin) continue;  // a bias
    const uint32_t q = k / cin, ci = k - q * cin, co = q / 9u, tap = q - co * 9u;
    const __nv_bfloat16 h = __float2bfloat16_rn(wi);
    t.wf[l][((size_t)((ci >> 3) * 9 + tap) * cout + co) * 8 + (ci & 7)] = h;
    t.wa[l][((size_t)((co >> 3) * 9 + (8 - tap)) * cin + ci) * 8 + (co & 7)] = h;
  }
}

// Weights in the operand order of the tensor-core convolution (k_conv.cu):
// wm[ci / 8][tap][co][ci % 8], i.e. for every 8-channel input group and tap a
// column of 16-byte rows, one per output channel.  wf: the forward operator
// from w[co][tap][ci].  wa: the adjoint (input gradient of a 3x3 'same'
// convolution), the operator with C_in' = cout, C_out' = cin and weights
// w'[ci][tap][co] = w[co][8 - tap][ci], in the same order:
// wa[co / 8][tap][ci][co % 8].  Either output may be null.
template <class T>
__global__ void k_pack_weights(const T* __restrict__ w, int cout, int cin, __nv_bfloat16* __restrict__ wf,
                               __nv_bfloat16* __restrict__ wa) {
  const size_t n = (size_t)cout * 9 * cin;
  for (size_t i = gtid(); i < n; i += gstride()) {
    const int ci = (int)(i % cin);
    const size_t t = i / cin;
    const int tap = (int)(t % 9), co = (int)(t / 9);
    const __nv_bfloat16 v = to_bf(w[i]);
    if (wf) wf[(((size_t)(ci >> 3) * 9 + tap) * cout + co) * 8 + (ci & 7)] = v;
    if (wa) wa[(((size_t)(co >> 3) * 9 + (8 - tap)) * cin + ci) * 8 + (co & 7)] = v;
  }
}

}  // namespace

#define NN_LAUNCH(kernel, n, ...)                                \
  do {                                                           \
    kernel<<<blocks_for(n), 256, 0, s>>>(__VA_ARGS__);           \
    return cudaGetLastError();                                   \
  } while (0)

cudaError_t image_mean(const float* img, int n, int hw, float* scale, cudaStream_t s) {
  k_image_mean<<<n, 256, 0, s>>>(img, hw, scale);
  return cudaGetLastError();
}
cudaError_t pack_input(const float* img, const float* scale, int n, int hw, __nv_bfloat16* x, cudaStream_t s) {
  NN_LAUNCH(k_pack_input, (size_t)n * hw, img, scale, n, hw, x);
}
cudaError_t unpack_output(const float* img, const float* scale, const float* net, int n, int hw, float* out,
                          cudaStream_t s) {
  NN_LAUNCH(k_unpack_output, (size_t)n * hw, img, scale, net, n, hw, out);
}
cudaError_t mse(const float* img, const float* tgt, const float* scale, const float* net, int n, int hw,
                __nv_bfloat16* gb, float* db, double* loss, cudaStream_t s) {
  NN_LAUNCH(k_mse, (size_t)n * hw, img, tgt, scale, net, n, hw, reinterpret_cast<uint4*>(gb), db, loss);
}
cudaError_t mask(MaskMode mode, const float* g, const float* gp, const __nv_bfloat16* y, int n, int h, int w, int c,
                 __nv_bfloat16* gb, float* db, cudaStream_t s) {
  // the thread layout needs 8 .. 32 eight-channel groups to divide a block
  if (c < 16 || c > 256 || (c & (c - 1))) return cudaErrorInvalidValue;
  const size_t npix = (size_t)n * h * w, items = mode == MASK_POOL ? npix / 4 : npix;
  const size_t blocks = (items * (c / 8) + kMaskThreads - 1) / kMaskThreads;
  const int grid = (int)(blocks < 152 * 8 ? blocks : 152 * 8);
  const uint4* yq = reinterpret_cast<const uint4*>(y);
  uint4* gq = reinterpret_cast<uint4*>(gb);
  if (mode == MASK_PLAIN) k_mask<0><<<grid, kMaskThreads, 0, s>>>(g, gp, yq, npix, h, w, c, gq, db);
  else if (mode == MASK_UP) k_mask<1><<<grid, kMaskThreads, 0, s>>>(g, gp, yq, npix, h, w, c, gq, db);
  else k_mask<2><<<grid, kMaskThreads, 0, s>>>(g, gp, yq, npix, h, w, c, gq, db);
  return cudaGetLastError();
}
cudaError_t pool_fwd(const __nv_bfloat16* x, int n, int h, int w, int c, __nv_bfloat16* y, cudaStream_t s) {
  k_pool_fwd<<<n * (h / 2), 256, 0, s>>>(reinterpret_cast<const uint4*>(x), w, c / 8, reinterpret_cast<uint4*>(y));
  return cudaGetLastError();
}
cudaError_t up_concat(const __nv_bfloat16* x, const __nv_bfloat16* skip, int n, int h, int w, int c, int cs,
                      __nv_bfloat16* y, cudaStream_t s) {
  k_up_concat<<<n * 2 * h, 256, 0, s>>>(reinterpret_cast<const uint4*>(x), reinterpret_cast<const uint4*>(skip), h, w,
                                        c / 8, cs / 8, reinterpret_cast<uint4*>(y));
  return cudaGetLastError();
}
cudaError_t adam(float* w, const float* g, float* m, float* v, const LayerTable& t, float lr, int step, cudaStream_t s) {
  const float b1 = 0.9f, b2 = 0.999f;
  const float c1 = 1.f - powf(b1, (float)step), c2 = 1.f - powf(b2, (float)step);
  NN_LAUNCH(k_adam, (size_t)t.begin[t.layers], w, g, m, v, t, lr, b1, b2, 1e-8f, c1, c2);
}
cudaError_t pack_weights(const float* w, int cout, int cin, __nv_bfloat16* wf, __nv_bfloat16* wa, cudaStream_t s) {
  NN_LAUNCH(k_pack_weights<float>, (size_t)cout * 9 * cin, w, cout, cin, wf, wa);
}
cudaError_t pack_weights_bf16(const __nv_bfloat16* w, int cout, int cin, __nv_bfloat16* wf, cudaStream_t s) {
  NN_LAUNCH(k_pack_weights<__nv_bfloat16>, (size_t)cout * 9 * cin, w, cout, cin, wf, nullptr);
}

}  // namespace nn
}  // namespace mcx

// FDK pre-weighting and ramp filtering of detector rows by fast Fourier
// transforms (arXiv 2201.13191 Sec. II-E; the direct sum and its kernel h are in
// k_recon.cu):
//   q(u_i) = du sum_j h(i - j) x_j,  x_j = w(u_j, v) p(u_j).
//
// Summed by parts, sum_j h(i - j) x_j = sum_j G(i - j) (x_j - x_{j-1}) with
// G(n) = sum_{m <= n} h(m) and x zero outside the row.  The ramp takes the
// smooth part of a row away again; a transform of the row itself would leave
// its rounding (2^-24 of the largest x) in the result, a transform of the
// differences leaves 2^-24 of the largest difference.  Two rows are the real
// and imaginary part of one transform of N >= 2 nu points.
//
// One thread holds 16 points.  A level takes the points n + k M of a block of
// length R M (R = 16, the last level the remaining factor), transforms them in
// registers and leaves them, times W^(n q), in the places they came from:
// block q of the next level.  So every level reads and writes a thread's own
// places of one shared array, the frequencies end in digit-reversed places, and
// the inverse walks the same levels back; multiplying by the kernel's spectrum
// happens in registers between the two.  368640 rows of 1024: 2.4 ms (1.26 TB/s
// read and written, bound by issue slots) against 31.9 ms of direct sums.
#include <stdint.h>

#include "mc_internal.h"

namespace mcx {
namespace {

template <int LOGN>
struct Plan {
  static constexpr int N = 1 << LOGN;
  static constexpr int T = N / 16;                      // threads per transform
  static constexpr int threads = T < 128 ? 128 : T;
  static constexpr int per_block = threads / T;         // transforms per block
  static constexpr int levels = (LOGN + 3) / 4;
  static constexpr int slot = N + N / 16;               // padded points of one transform in shared memory
  __host__ __device__ static constexpr int logr(int l) { return LOGN - 4 * l < 4 ? LOGN - 4 * l : 4; }
};

__device__ __forceinline__ float2 cmul(float2 a, float2 b) {
  return make_float2(fmaf(a.x, b.x, -a.y * b.y), fmaf(a.x, b.y, a.y * b.x));
}
__device__ __forceinline__ float2 cadd(float2 a, float2 b) { return make_float2(a.x + b.x, a.y + b.y); }
__device__ __forceinline__ float2 csub(float2 a, float2 b) { return make_float2(a.x - b.x, a.y - b.y); }
// a times exp(-i phi) (INV: exp(+i phi)) for cos and sin of phi
template <bool INV>
__device__ __forceinline__ float2 crot(float2 a, float c, float s) {
  return INV ? make_float2(fmaf(a.x, c, -a.y * s), fmaf(a.x, s, a.y * c))
             : make_float2(fmaf(a.x, c, a.y * s), fmaf(a.y, c, -a.x * s));
}

// Discrete Fourier transform of R points in natural order, in registers.
template <int R, bool INV>
__device__ __forceinline__ void dft(float2 (&v)[R]) {
  if constexpr (R == 2) {
    const float2 a = v[0];
    v[0] = cadd(a, v[1]);
    v[1] = csub(a, v[1]);
  } else if constexpr (R > 2) {
    float2 e[R / 2], o[R / 2];
#pragma unroll
    for (int k = 0; k < R / 2; ++k) {
      e[k] = v[2 * k];
      o[k] = v[2 * k + 1];
    }
    dft<R / 2, INV>(e);
    dft<R / 2, INV>(o);
    // cos and sin of 2 pi k / 16
    constexpr float kC[8] = {1.f, 0.92387953251f, 0.70710678119f, 0.38268343236f,
                             0.f, -0.38268343236f, -0.70710678119f, -0.92387953251f};
    constexpr float kS[8] = {0.f, 0.38268343236f, 0.70710678119f, 0.92387953251f,
                             1.f, 0.92387953251f, 0.70710678119f, 0.38268343236f};
#pragma unroll
    for (int k = 0; k < R / 2; ++k) {
      constexpr int step = 16 / R;
      float2 t = o[k];
      if (k * step == 4) t = INV ? make_float2(-o[k].y, o[k].x) : make_float2(o[k].y, -o[k].x);
      else if (k > 0) t = crot<INV>(o[k], kC[k * step], kS[k * step]);
      v[k] = cadd(e[k], t);
      v[k + R / 2] = csub(e[k], t);
    }
  }
}

// v[q] *= w^q for q = 1 .. R - 1 (conjugate powers where INV), by a tree of products.
template <int R, bool INV>
__device__ __forceinline__ void twiddle(float2 (&v)[R], float2 w) {
  if (INV) w.y = -w.y;
  float2 p[R];
  p[0] = make_float2(1.f, 0.f);
  p[1] = w;
#pragma unroll
  for (int q = 2; q < R; ++q) p[q] = cmul(p[q / 2], p[q - q / 2]);
#pragma unroll
  for (int q = 1; q < R; ++q) v[q] = cmul(v[q], p[q]);
}

__device__ __forceinline__ int padded(int p) { return p + (p >> 4); }

// Level l >= 1 of the transform in `sh` (this transform's slot), thread t.
// FWD: butterfly then twiddle; inverse: twiddle then butterfly.  On the last
// level the spectrum `g` ([e T + t], e the point's number in the thread) is
// multiplied in and the level is undone in registers; with `out` set the
// frequencies are written there instead (making the spectrum itself).
template <int LOGN, int L, bool INV>
__device__ __forceinline__ void level(float2* sh, int t, const float2* __restrict__ tw, const float2* __restrict__ g,
                                      float2* out) {
  using P = Plan<LOGN>;
  constexpr int LR = P::logr(L), R = 1 << LR, len = P::N >> (4 * L), M = len >> LR;
  constexpr bool last = L == P::levels - 1;
#pragma unroll
  for (int j = 0; j < 16 / R; ++j) {
    const int b = t + j * P::T, s = b / M, n = b - s * M, base = s * len + n;
    float2 v[R];
#pragma unroll
    for (int k = 0; k < R; ++k) v[k] = sh[padded(base + k * M)];
    if constexpr (last) {
      dft<R, false>(v);
      if (out) {
#pragma unroll
        for (int k = 0; k < R; ++k) out[(j * R + k) * P::T + t] = v[k];
      } else {
#pragma unroll
        for (int k = 0; k < R; ++k) v[k] = cmul(v[k], __ldg(g + (j * R + k) * P::T + t));
        dft<R, true>(v);
      }
    } else {
      const float2 w = __ldg(tw + n * (P::N / len));
      if (INV) {
        twiddle<R, true>(v, w);
        dft<R, true>(v);
      } else {
        dft<R, false>(v);
        twiddle<R, false>(v, w);
      }
    }
#pragma unroll
    for (int k = 0; k < R; ++k) sh[padded(base + k * M)] = v[k];
  }
}

template <int LOGN>
__device__ __forceinline__ void middle(float2* sh, int t, const float2* tw, const float2* g, float2* out) {
  constexpr int n = Plan<LOGN>::levels;  // 2 .. 4
  __syncthreads();
  level<LOGN, 1, false>(sh, t, tw, g, out);
  if constexpr (n > 2) {
    __syncthreads();
    level<LOGN, 2, false>(sh, t, tw, g, out);
  }
  if constexpr (n > 3) {
    __syncthreads();
    level<LOGN, 3, false>(sh, t, tw, g, out);
    __syncthreads();
    level<LOGN, 2, true>(sh, t, tw, g, out);
  }
  if constexpr (n > 2) {
    __syncthreads();
    level<LOGN, 1, true>(sh, t, tw, g, out);
  }
  __syncthreads();
}

// W^k = exp(-2 pi i k / N)
__global__ void k_ramp_twiddles(int n, float2* __restrict__ tw) {
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= n) return;
  float s, c;
  sincospif(2.f * (float)k / (float)n, &s, &c);
  tw[k] = make_float2(c, -s);
}

// The spectrum of G (N values: G(n) at n mod N), in the order level() reads it.
template <int LOGN>
__global__ void __launch_bounds__(Plan<LOGN>::threads) k_ramp_spectrum(const float* __restrict__ g, float scale,
                                                                       const float2* __restrict__ tw,
                                                                       float2* __restrict__ out) {
  using P = Plan<LOGN>;
  extern __shared__ float2 sh_all[];
  const int t = threadIdx.x % P::T;
  float2* sh = sh_all + (threadIdx.x / P::T) * P::slot;  // every transform of the block makes the same values
  float2 v[16];
#pragma unroll
  for (int k = 0; k < 16; ++k) v[k] = make_float2(g[t + k * P::T] * scale, 0.f);
  dft<16, false>(v);
  twiddle<16, false>(v, __ldg(tw + t));
#pragma unroll
  for (int k = 0; k < 16; ++k) sh[padded(t + k * P::T)] = v[k];
  middle<LOGN>(sh, t, tw, nullptr, out);
}

// Filters rows 2 b and 2 b + 1 (b the transform's number).  A row holding a
// value that is not finite (or close to overflow) would spoil the other one:
// it enters as zeros and its outputs are summed directly.
template <int LOGN>
__global__ void __launch_bounds__(Plan<LOGN>::threads) k_ramp_filter(const float* __restrict__ p, int nu, int nv,
                                                                     int rows, float du, float dv, float sod,
                                                                     const float2* __restrict__ tw,
                                                                     const float2* __restrict__ g,
                                                                     float* __restrict__ q) {
  using P = Plan<LOGN>;
  extern __shared__ float2 sh_all[];
  __shared__ int bad[2 * P::per_block];
  const int f = threadIdx.x / P::T, t = threadIdx.x % P::T;
  float2* sh = sh_all + f * P::slot;
  const int r0 = 2 * (blockIdx.x * P::per_block + f);
  if (threadIdx.x < 2 * P::per_block) bad[threadIdx.x] = 0;
  __syncthreads();
  const float va = ((float)(r0 % nv) - 0.5f * (float)(nv - 1)) * dv;
  const float vb = ((float)((r0 + 1) % nv) - 0.5f * (float)(nv - 1)) * dv;
  const float* pa = p + (size_t)r0 * nu;
  const bool has_b = r0 + 1 < rows;
  // the weighted value, as the direct sum takes it
  auto weighted = [&](float x, float vv, int i) -> float {
    const float uu = ((float)i - 0.5f * (float)(nu - 1)) * du;
    return x * sod * rsqrtf(sod * sod + uu * uu + vv * vv);
  };
  float2 v[16];
  if (r0 < rows) {
#pragma unroll
    for (int k = 0; k < 16; ++k) {
      const int i = t + k * P::T;
      v[k] = make_float2(i < nu ? __ldg(pa + i) : 0.f, i < nu && has_b ? __ldg(pa + nu + i) : 0.f);
    }
  }
  bool bad_a = false, bad_b = false;
#pragma unroll
  for (int k = 0; k < 16; ++k) {
    const int i = t + k * P::T;
    v[k] = r0 < rows && i < nu ? make_float2(weighted(v[k].x, va, i), weighted(v[k].y, vb, i)) : make_float2(0.f, 0.f);
    bad_a |= !(fabsf(v[k].x) < 1e30f);
    bad_b |= !(fabsf(v[k].y) < 1e30f);
    sh[padded(i)] = v[k];
  }
  if (bad_a) bad[2 * f] = 1;
  if (bad_b) bad[2 * f + 1] = 1;
  __syncthreads();
  bad_a = bad[2 * f] != 0;
  bad_b = bad[2 * f + 1] != 0;
#pragma unroll
  for (int k = 0; k < 16; ++k) {
    const int i = t + k * P::T;
    if (i > 0) v[k] = csub(v[k], sh[padded(i - 1)]);
    if (bad_a) v[k].x = 0.f;
    if (bad_b) v[k].y = 0.f;
  }
  __syncthreads();
  dft<16, false>(v);
  const float2 w = __ldg(tw + t);
  twiddle<16, false>(v, w);
#pragma unroll
  for (int k = 0; k < 16; ++k) sh[padded(t + k * P::T)] = v[k];
  middle<LOGN>(sh, t, tw, g, nullptr);
#pragma unroll
  for (int k = 0; k < 16; ++k) v[k] = sh[padded(t + k * P::T)];
  twiddle<16, true>(v, w);
  dft<16, true>(v);
  const float h0 = 0.25f / (du * du), c = 1.f / (9.8696044f * du * du);
#pragma unroll
  for (int row = 0; row < 2; ++row) {
    const int r = r0 + row;
    if (r >= rows) continue;
    const bool direct = row ? bad_b : bad_a;
#pragma unroll
    for (int k = 0; k < 16; ++k) {
      const int i = t + k * P::T;
      if (i >= nu) continue;
      float o = row ? v[k].y : v[k].x;
      if (direct) {
        float acc = 0.f;
        for (int j = 0; j < nu; ++j) {
          const int d = i - j;
          const float h = d == 0 ? h0 : ((d & 1) ? -c / ((float)d * (float)d) : 0.f);
          acc = fmaf(weighted(__ldg(p + (size_t)r * nu + j), row ? vb : va, j), h, acc);
        }
        o = acc * du;
      }
      q[(size_t)r * nu + i] = o;
    }
  }
}

template <int LOGN>
cudaError_t launch(const float* p, int nu, int nv, int rows, float du, float dv, float sod, float* ramp, float* q,
                   bool tables, cudaStream_t s) {
  using P = Plan<LOGN>;
  const int smem = P::per_block * P::slot * (int)sizeof(float2);
  if (smem > 48 * 1024) {
    cudaError_t e = cudaFuncSetAttribute(k_ramp_filter<LOGN>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e == cudaSuccess)
      e = cudaFuncSetAttribute(k_ramp_spectrum<LOGN>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e != cudaSuccess) return e;
  }
  float2 *tw = reinterpret_cast<float2*>(ramp + P::N), *spec = tw + P::N;
  if (tables) {
    k_ramp_twiddles<<<(P::N + 255) / 256, 256, 0, s>>>(P::N, tw);
    k_ramp_spectrum<LOGN><<<1, P::threads, smem, s>>>(ramp, du / (float)P::N, tw, spec);
  }
  const int pairs = (rows + 1) / 2;
  k_ramp_filter<LOGN><<<(pairs + P::per_block - 1) / P::per_block, P::threads, smem, s>>>(p, nu, nv, rows, du, dv, sod,
                                                                                          tw, spec, q);
  return cudaGetLastError();
}

}  // namespace

int ramp_points(int nu) {
  if (nu > 4096) return 0;
  int n = 256;
  while (n < 2 * nu) n <<= 1;
  return n;
}

// G(n) = sum_{m <= n} h(m), n = -nu .. nu - 1, at n mod N: the taps in FP32, as the direct sum takes them, added in
// FP64.
void ramp_kernel(int nu, float du, float* g) {
  const int n = ramp_points(nu);
  for (int i = 0; i < n; ++i) g[i] = 0.f;
  const float h0 = 0.25f / (du * du), c = 1.f / (9.8696044f * du * du);
  double sum = 0.0;
  for (int m = -(nu - 1); m <= nu - 1; ++m) {
    const float d = (float)m;
    sum += m == 0 ? h0 : ((m & 1) ? -c / (d * d) : 0.f);
    g[m & (n - 1)] = (float)sum;
  }
}

cudaError_t ramp_filter(const float* p, int nu, int nv, int rows, float du, float dv, float sod, float* ramp, float* q,
                        bool tables, cudaStream_t s) {
  switch (ramp_points(nu)) {
    case 256: return launch<8>(p, nu, nv, rows, du, dv, sod, ramp, q, tables, s);
    case 512: return launch<9>(p, nu, nv, rows, du, dv, sod, ramp, q, tables, s);
    case 1024: return launch<10>(p, nu, nv, rows, du, dv, sod, ramp, q, tables, s);
    case 2048: return launch<11>(p, nu, nv, rows, du, dv, sod, ramp, q, tables, s);
    case 4096: return launch<12>(p, nu, nv, rows, du, dv, sod, ramp, q, tables, s);
    case 8192: return launch<13>(p, nu, nv, rows, du, dv, sod, ramp, q, tables, s);
  }
  return cudaErrorInvalidValue;
}

}  // namespace mcx

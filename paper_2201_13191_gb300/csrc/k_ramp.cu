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
// happens in registers between the two.  368640 rows of 1024: 2.0 ms (1.5 TB/s
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

// W^k = exp(-2 pi i k / N), and the taps h(d) at d mod N, as the direct sum takes them
__global__ void k_ramp_twiddles(int n, float du, float2* __restrict__ tw, float* __restrict__ taps) {
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= n) return;
  const int d = min(k, n - k);
  taps[k] = d == 0 ? 0.25f / (du * du) : ((d & 1) ? -(1.f / (9.8696044f * du * du)) / ((float)d * (float)d) : 0.f);
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

// The weighted value of pixel i of a row at height v, as the direct sum takes it.
__device__ __forceinline__ float weighted(float x, float v, int i, int nu, float du, float sod) {
  const float u = ((float)i - 0.5f * (float)(nu - 1)) * du;
  return x * sod * rsqrtf(sod * sod + u * u + v * v);
}

// A transform rounds every output to the size of its largest difference; a direct sum rounds each term to its own.  The
// two agree (a few units of 2^-24 of the row's values) while no difference stands out.  Differences above
// 3 mean|x| + 6 mean|d| are therefore left out of the transform and added with their taps G(i - j), and pixels above
// kPixel times mean|x| (or not finite) with the taps h(i - j), whose zeros and 1 / n^2 keep such a pixel in its place.
// There can be few of either (their share of the sums), and a row of noise, or of an object that fills a sixth of it, has
// none.  Rows whose sums differ in their binary exponent are brought to one size (powers of two), since the two rows of a
// transform share its rounding.
constexpr float kPixel = 16.f;
constexpr float kHuge = 1e30f;

template <int LOGN>
struct Large {
  static constexpr int words = Plan<LOGN>::N / 64 + 1;  // nu + 1 bits
  uint32_t pixel[2][words], step[2][words];             // of the transform's two rows
};

// Of a transform's two rows: sum of |x|, sum and largest of |d| (its bits: above infinity's where it is no number).
struct RowSize {
  float2 x, d;
  uint32_t ma, mb;
  __device__ __forceinline__ void add(float2 dd) {
    d.x += fabsf(dd.x);
    d.y += fabsf(dd.y);
    ma = max(ma, __float_as_uint(dd.x) & 0x7FFFFFFFu);
    mb = max(mb, __float_as_uint(dd.y) & 0x7FFFFFFFu);
  }
  // Largest ordinary difference; the rows of few pixels have few to take a mean of.
  __device__ __forceinline__ float2 limit(int nu) const {
    const float n = 3.f / (float)nu, m = 6.f / (float)(nu + 64);
    return make_float2(fmaf(n, x.x, m * d.x), fmaf(n, x.y, m * d.y));
  }
};

// Over a transform's threads; a barrier of the block lies between what its threads wrote before and what they read
// afterwards.
template <int LOGN>
__device__ __forceinline__ RowSize row_size(RowSize s, RowSize* part, int t) {
  constexpr int T = Plan<LOGN>::T, seg = T < 32 ? T : 32;
#pragma unroll
  for (int o = seg / 2; o > 0; o >>= 1) {
    s.x.x += __shfl_xor_sync(0xffffffffu, s.x.x, o);
    s.x.y += __shfl_xor_sync(0xffffffffu, s.x.y, o);
    s.d.x += __shfl_xor_sync(0xffffffffu, s.d.x, o);
    s.d.y += __shfl_xor_sync(0xffffffffu, s.d.y, o);
  }
  const uint32_t lanes = seg == 32 ? 0xffffffffu : 0xffffu << (threadIdx.x & 16);
  s.ma = __reduce_max_sync(lanes, s.ma);
  s.mb = __reduce_max_sync(lanes, s.mb);
  if (t % seg == 0) part[t / seg] = s;
  __syncthreads();
  s = part[0];
#pragma unroll
  for (int i = 1; i < T / seg; ++i) {
    s.x = cadd(s.x, part[i].x);
    s.d = cadd(s.d, part[i].d);
    s.ma = max(s.ma, part[i].ma);
    s.mb = max(s.mb, part[i].mb);
  }
  return s;
}

// Marks the large pixels and differences of the rows in sh (weighted values, whose sums of |x| are `sum`) and leaves the
// differences without them there, each thread its own places; returns the sums of |x| without the large pixels.  All
// threads of the block call it.
template <int LOGN>
__device__ __noinline__ float2 take_large(float2* sh, Large<LOGN>* large, RowSize* part, float2 sum, int nu, int t) {
  constexpr int T = Plan<LOGN>::T, words = Large<LOGN>::words;
  uint32_t* const mark = &large->pixel[0][0];
  for (int i = t; i < 4 * words; i += T) mark[i] = 0u;
  __syncthreads();
  const float n = (float)nu;
  for (;;) {  // every round but the last takes a pixel at least
    const float la = sum.x < kHuge ? kPixel * sum.x : 0.1f * kHuge * n, lb = sum.y < kHuge ? kPixel * sum.y : 0.1f * kHuge * n;
    bool took = false;
    RowSize s = {};
#pragma unroll 1
    for (int k = 0; k < 16; ++k) {
      const int i = t + k * T;
      float2 x = sh[padded(i)];
      if (!(fabsf(x.x) * n <= la)) {
        atomicOr(&large->pixel[0][i >> 5], 1u << (i & 31));
        x.x = 0.f;
        took = true;
      }
      if (!(fabsf(x.y) * n <= lb)) {
        atomicOr(&large->pixel[1][i >> 5], 1u << (i & 31));
        x.y = 0.f;
        took = true;
      }
      sh[padded(i)] = x;
      s.x = cadd(s.x, make_float2(fabsf(x.x), fabsf(x.y)));
    }
    took = __syncthreads_or(took);
    sum = row_size<LOGN>(s, part, t).x;
    if (!took) break;
  }
  float2 d[16];
  RowSize s = {};
#pragma unroll
  for (int k = 0; k < 16; ++k) {
    const int i = t + k * T;
    d[k] = sh[padded(i)];
    if (i > 0) d[k] = csub(d[k], sh[padded(i - 1)]);
    s.add(d[k]);
  }
  __syncthreads();
  s = row_size<LOGN>(s, part, t);
  s.x = sum;
  const float2 lim = s.limit(nu);
#pragma unroll
  for (int k = 0; k < 16; ++k) {
    const int i = t + k * T;
    if (fabsf(d[k].x) > lim.x) {
      atomicOr(&large->step[0][i >> 5], 1u << (i & 31));
      d[k].x = 0.f;
    }
    if (fabsf(d[k].y) > lim.y) {
      atomicOr(&large->step[1][i >> 5], 1u << (i & 31));
      d[k].y = 0.f;
    }
    sh[padded(i)] = d[k];
  }
  return sum;
}

// Adds what the large pixels and differences of a row (p, at height v) contribute to the outputs that this thread stored
// in q; gs, hs: G(d) and h(d) at d mod N (one load and one multiply-add per tap: an object 50 pixels wide, whose every
// pixel is a large one, costs as much again as the transform).
template <int LOGN>
__device__ __noinline__ void add_large(const float* __restrict__ p, float* __restrict__ q, const uint32_t* pixel,
                                       const uint32_t* step, const float* __restrict__ gs,
                                       const float* __restrict__ hs, int nu, float du, float v, float sod, int t) {
  using P = Plan<LOGN>;
  uint32_t any = 0u;
  for (int k = 0; k < Large<LOGN>::words; ++k) any |= pixel[k] | step[k];
  if (!any) return;
  float acc[16] = {};
  bool nan = false;  // then so is every output
  for (int b = 0; b < Large<LOGN>::words && !nan; ++b) {
    for (uint32_t m = pixel[b]; m && !nan; m &= m - 1) {
      const int j = 32 * b + __ffs(m) - 1;
      const float x = weighted(__ldg(p + j), v, j, nu, du, sod);
#pragma unroll
      for (int k = 0; k < 16; ++k) acc[k] = fmaf(x, __ldg(hs + ((t + k * P::T - j) & (P::N - 1))), acc[k]);
      nan = x != x;
    }
    for (uint32_t m = nan ? 0u : step[b]; m; m &= m - 1) {
      const int j = 32 * b + __ffs(m) - 1;
      auto at = [&](int i) -> float {  // the row without its large pixels
        return i < 0 || i >= nu || ((pixel[i >> 5] >> (i & 31)) & 1u) ? 0.f : weighted(__ldg(p + i), v, i, nu, du, sod);
      };
      const float x = at(j) - at(j - 1);
#pragma unroll
      for (int k = 0; k < 16; ++k) acc[k] = fmaf(x, __ldg(gs + ((t + k * P::T - j) & (P::N - 1))), acc[k]);
    }
  }
#pragma unroll
  for (int k = 0; k < 16; ++k) {
    const int i = t + k * P::T;
    if (i < nu) q[i] = fmaf(acc[k], du, q[i]);
  }
}

// Filters rows 2 b and 2 b + 1 (b the transform's number); ramp: G, then tw, the spectrum g and the taps.
template <int LOGN>
__global__ void __launch_bounds__(Plan<LOGN>::threads) k_ramp_filter(const float* __restrict__ p, int nu, int nv,
                                                                     int rows, float du, float dv, float sod,
                                                                     const float* __restrict__ ramp,
                                                                     const float2* __restrict__ tw,
                                                                     const float2* __restrict__ g,
                                                                     float* __restrict__ q) {
  using P = Plan<LOGN>;
  extern __shared__ float2 sh_all[];
  __shared__ RowSize part[P::per_block][P::T < 32 ? 1 : P::T / 32];
  __shared__ Large<LOGN> large[P::per_block];
  const int f = threadIdx.x / P::T, t = threadIdx.x % P::T;
  float2* sh = sh_all + f * P::slot;
  const int r0 = 2 * (blockIdx.x * P::per_block + f);
  const float va = ((float)(r0 % nv) - 0.5f * (float)(nv - 1)) * dv;
  const float vb = ((float)((r0 + 1) % nv) - 0.5f * (float)(nv - 1)) * dv;
  const float* pa = p + (size_t)r0 * nu;
  const bool has_b = r0 + 1 < rows;
  float2 v[16];
  if (r0 < rows) {
#pragma unroll
    for (int k = 0; k < 16; ++k) {
      const int i = t + k * P::T;
      v[k] = make_float2(i < nu ? __ldg(pa + i) : 0.f, i < nu && has_b ? __ldg(pa + nu + i) : 0.f);
    }
  }
  RowSize size = {};
#pragma unroll
  for (int k = 0; k < 16; ++k) {
    const int i = t + k * P::T;
    v[k] = r0 < rows && i < nu ? make_float2(weighted(v[k].x, va, i, nu, du, sod), weighted(v[k].y, vb, i, nu, du, sod))
                               : make_float2(0.f, 0.f);
    size.x = cadd(size.x, make_float2(fabsf(v[k].x), fabsf(v[k].y)));
    sh[padded(i)] = v[k];
  }
  __syncthreads();
#pragma unroll
  for (int k = 0; k < 16; ++k) {
    const int i = t + k * P::T;
    if (i > 0) v[k] = csub(v[k], sh[padded(i - 1)]);
    size.add(v[k]);
  }
  size = row_size<LOGN>(size, part[f], t);
  const float2 lim = size.limit(nu);
  const bool mine = !(__uint_as_float(size.ma) <= lim.x && __uint_as_float(size.mb) <= lim.y && size.x.x < kHuge && size.x.y < kHuge);
  const bool with_large = P::per_block > 1 ? __syncthreads_or(mine) : mine;
  float2 sum = size.x;
  if (with_large) {
    sum = take_large<LOGN>(sh, large + f, part[f], sum, nu, t);
#pragma unroll
    for (int k = 0; k < 16; ++k) v[k] = sh[padded(t + k * P::T)];
  }
  const int ea = max(__float_as_int(sum.x) >> 23, 1), eb = max(__float_as_int(sum.y) >> 23, 1);
  if (ea != eb || sum.x == 0.f || sum.y == 0.f) {
    const float fa = __int_as_float((254 - ea) << 23), fb = __int_as_float((254 - eb) << 23);
#pragma unroll
    for (int k = 0; k < 16; ++k) v[k] = make_float2(v[k].x * fa, v[k].y * fb);
  }
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
  if (ea != eb || sum.x == 0.f || sum.y == 0.f) {  // an empty row stays empty
    const float fa = sum.x == 0.f ? 0.f : __int_as_float(ea << 23), fb = sum.y == 0.f ? 0.f : __int_as_float(eb << 23);
#pragma unroll
    for (int k = 0; k < 16; ++k) v[k] = make_float2(v[k].x * fa, v[k].y * fb);
  }
#pragma unroll
  for (int row = 0; row < 2; ++row) {
    const int r = r0 + row;
    if (r >= rows) continue;
#pragma unroll
    for (int k = 0; k < 16; ++k) {
      const int i = t + k * P::T;
      if (i < nu) q[(size_t)r * nu + i] = row ? v[k].y : v[k].x;
    }
    if (with_large)
      add_large<LOGN>(p + (size_t)r * nu, q + (size_t)r * nu, large[f].pixel[row], large[f].step[row], ramp,
                      ramp + 5 * P::N, nu, du, row ? vb : va, sod, t);
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
    k_ramp_twiddles<<<(P::N + 255) / 256, 256, 0, s>>>(P::N, du, tw, ramp + 5 * P::N);
    k_ramp_spectrum<LOGN><<<1, P::threads, smem, s>>>(ramp, du / (float)P::N, tw, spec);
  }
  const int pairs = (rows + 1) / 2;
  k_ramp_filter<LOGN><<<(pairs + P::per_block - 1) / P::per_block, P::threads, smem, s>>>(p, nu, nv, rows, du, dv, sod,
                                                                                          ramp, tw, spec, q);
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

// Iterative scatter correction plumbing (arXiv 2201.13191 Sec. II-E, Fig.
// flowchart, eq. Correction): conversion of intensities to line integrals,
// FDK (cone-beam filtered backprojection) for the circular orbit of this
// library's geometry, multi-level Otsu segmentation, conversion of the
// segmented volume to material ids and densities, its 2x2x2 down-sampling for
// the Monte Carlo step (Sec. II-C.2), and the correction
// c = a - ln(Ip / (Ip + Is)).
#include <cuda_fp16.h>
#include <stdint.h>

#include "mc_internal.h"

namespace mcx {
namespace {

__device__ __forceinline__ size_t gtid() { return (size_t)blockIdx.x * blockDim.x + threadIdx.x; }
__device__ __forceinline__ size_t gstride() { return (size_t)gridDim.x * blockDim.x; }
int blocks_for(size_t n) {
  const size_t b = (n + 255) / 256;
  return (int)(b < 152 * 32 ? (b > 0 ? b : 1) : 152 * 32);
}

// a = -ln(I / I0) per pixel (I0 is one flat-field image shared by all projections).
__global__ void k_log_norm(const float* __restrict__ I, const float* __restrict__ I0, size_t img, size_t n,
                           float* __restrict__ a) {
  for (size_t i = gtid(); i < n; i += gstride()) {
    const float v = fmaxf(I[i], 1e-30f), f = fmaxf(I0[i % img], 1e-30f);
    a[i] = -logf(v / f);
  }
}

// FDK pre-weighting and ramp filtering of detector rows:
//   q(u_i) = du * sum_j h(i - j) * w(u_j, v) p(u_j),  w = D / sqrt(D^2 + u^2 + v^2)
// with u, v the pixel-centre offsets scaled to the isocentre plane, D = SOD,
// du the isocentre pixel pitch and h the discrete Ram-Lak kernel
// h(0) = 1/(4 du^2), h(odd n) = -1/(n pi du)^2, h(even n != 0) = 0.
// A block filters kFiltRows rows; a warp owns 256 consecutive outputs (8 per
// lane) of each of them.  Walking j, lane l needs the taps h(i0 + m - j),
// m = 0..7, i0 = 8 l + warp base: one step in j shifts that window by one, so
// the new first tap is the previous lane's last one (a shuffle) and only lane 0
// reads a tap from shared memory.  The taps are shared by the rows, so each
// tap register feeds kFiltRows x 8 FMAs.
constexpr int kFiltOut = 8;
constexpr int kFiltRows = 4;
constexpr int kFiltThreads = 256;

__global__ void __launch_bounds__(kFiltThreads) k_fdk_filter(const float* __restrict__ p, int nu, int nv, int rows_total,
                                                             float du_iso, float dv_iso, float sod,
                                                             float* __restrict__ q) {
  extern __shared__ float fsh[];
  const int span = kFiltThreads * kFiltOut;               // outputs per pass of the block
  const int npad = (nu + span - 1) / span * span;
  const int H0 = npad + kFiltOut;                          // hs[d + H0] = h(d), |d| <= H0
  float* hs = fsh;
  float* rows = fsh + 2 * H0 + 1;                          // [kFiltRows][nu]
  const float h0 = 0.25f / (du_iso * du_iso), c = 1.f / (9.8696044f * du_iso * du_iso);
  for (int k = threadIdx.x; k <= 2 * H0; k += blockDim.x) {
    const int d = k - H0;
    hs[k] = d == 0 ? h0 : ((d & 1) ? -c / ((float)d * (float)d) : 0.f);
  }
  const int r0 = blockIdx.x * kFiltRows;
  for (int rr = 0; rr < kFiltRows; ++rr) {
    const int r = r0 + rr;
    const float vv = ((float)((r < rows_total ? r : 0) % nv) - 0.5f * (float)(nv - 1)) * dv_iso;
    for (int i = threadIdx.x; i < nu; i += blockDim.x) {
      const float uu = ((float)i - 0.5f * (float)(nu - 1)) * du_iso;
      rows[rr * nu + i] = r < rows_total ? p[(size_t)r * nu + i] * sod * rsqrtf(sod * sod + uu * uu + vv * vv) : 0.f;
    }
  }
  __syncthreads();
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  for (int base = warp * 256; base < npad; base += span) {
    const int i0 = base + lane * kFiltOut;
    float w[kFiltOut], acc[kFiltRows][kFiltOut];
#pragma unroll
    for (int m = 0; m < kFiltOut; ++m) {
      w[m] = hs[i0 + m + H0];
#pragma unroll
      for (int rr = 0; rr < kFiltRows; ++rr) acc[rr][m] = 0.f;
    }
#pragma unroll 4
    for (int j = 0; j < nu; ++j) {
#pragma unroll
      for (int rr = 0; rr < kFiltRows; ++rr) {
        const float x = rows[rr * nu + j];
#pragma unroll
        for (int m = 0; m < kFiltOut; ++m) acc[rr][m] = fmaf(x, w[m], acc[rr][m]);
      }
      const float carry = __shfl_up_sync(0xffffffffu, w[kFiltOut - 1], 1);
#pragma unroll
      for (int m = kFiltOut - 1; m > 0; --m) w[m] = w[m - 1];
      w[0] = lane == 0 ? hs[base - j - 1 + H0] : carry;
    }
#pragma unroll
    for (int rr = 0; rr < kFiltRows; ++rr) {
      const int r = r0 + rr;
      if (r >= rows_total) continue;
#pragma unroll
      for (int m = 0; m < kFiltOut; ++m)
        if (i0 + m < nu) q[(size_t)r * nu + i0 + m] = acc[rr][m] * du_iso;
    }
  }
}

// a / b, correctly rounded, from r = 1 / b (correctly rounded): the quotient a r
// corrected by its remainder (Markstein, IBM J. Res. Dev. 34, 1990).
__device__ __forceinline__ float div_by(float a, float b, float r) {
  const float q = a * r;
  return fmaf(fmaf(-q, b, a), r, q);
}

// Voxel-driven backprojection: f(x) = (dbeta / 2) sum_beta (D / (D - x.n))^2 q(u(x), v(x)),
// q bilinearly interpolated at the voxel's projection (zero outside the panel);
// the projections come in chunks, whose sums continue in vol (`first` starts
// them, `scale` is 1 until the last).  Each thread owns ZB voxels of one (x, y) column; per projection the
// source-side terms (depth, magnification, u and its bilinear weights) are
// computed once for the column, then each voxel adds its bilinear sample (the
// same expressions as one voxel at a time, so the same sums).  Bound by the L1
// wavefronts of the four taps (3.5 per load): a warp owns 8 x 4 columns, whose
// taps lie close together on the panel whatever the angle (a row of 32 in x
// spreads over up to 130 panel pixels).  256^3 x 360 projections of 1024^2: 15.3
// -> 9.3 ms with these tiles, the divisions by a stored reciprocal and ZB = 8.
// WIDE: projections of 2^31 pixels or more, or more than 2^22 rows, where a
// pixel's number needs 64 bits and its floor the conversion.
template <int ZB, bool WIDE>
__global__ void __launch_bounds__(256) k_fdk_backproject(const float* __restrict__ q, const float* __restrict__ cb,
                                                         const float* __restrict__ sb, int n_proj, int nu, int nv,
                                                         float du_iso, float dv_iso, float inv_du, float inv_dv,
                                                         float sod, int nx, int ny, int nz, float dx, float dy, float dz,
                                                         int first, float scale, float* __restrict__ vol) {
  // blocks of 16 x 16 columns (2 x 4 warps), x fastest, then y, then z
  const int bx_n = (nx + 15) / 16, by_n = (ny + 15) / 16;
  const int bx = (int)(blockIdx.x % (unsigned)bx_n);
  const unsigned byz = blockIdx.x / (unsigned)bx_n;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int ix = bx * 16 + (warp & 1) * 8 + (lane & 7);
  const int iy = (int)(byz % (unsigned)by_n) * 16 + (warp >> 1) * 4 + (lane >> 3);
  const int iz0 = (int)(byz / (unsigned)by_n) * ZB;
  if (ix >= nx || iy >= ny) return;
  const float x = ((float)ix - 0.5f * (float)(nx - 1)) * dx;
  const float y = ((float)iy - 0.5f * (float)(ny - 1)) * dy;
  const float cu = 0.5f * (float)(nu - 1), cv = 0.5f * (float)(nv - 1);
  const float u_top = (float)(nu - 1), v_top = (float)(nv - 1);
  constexpr float kFloor = 12582912.f;  // 1.5 x 2^23: a round-down add leaves floor in the low bits
  float z[ZB], acc[ZB];
#pragma unroll
  for (int j = 0; j < ZB; ++j) {
    z[j] = ((float)(iz0 + j) - 0.5f * (float)(nz - 1)) * dz;
    acc[j] = first || iz0 + j >= nz ? 0.f : vol[((size_t)(iz0 + j) * ny + iy) * nx + ix];
  }
  const size_t img = (size_t)nu * nv;
  // row v0 of q from column u0 on, v0 the floor fw of fv (a round-down add's sum where not WIDE)
  auto floor_of = [&](float f) { return WIDE ? floorf(f) : __fadd_rd(f, kFloor); };
  auto fraction = [&](float f, float fl) { return WIDE ? f - fl : f - (fl - kFloor); };
  auto whole = [&](float fl) { return WIDE ? (int)fl : __float_as_int(fl) - 0x4B400000; };
  auto row = [&](float fw, int u0) -> const float* {
    if constexpr (WIDE) return q + ((size_t)whole(fw) * nu + u0);
    else return q + (whole(fw) * nu + u0);
  };
#pragma unroll 1
  for (int k = 0; k < n_proj; ++k, q += img) {
    const float c = __ldg(cb + k), s = __ldg(sb + k);
    const float depth = sod - (x * c + y * s);  // distance from the source along the central ray
    const float mag = sod / depth;
    const float u = (-x * s + y * c) * mag;     // isocentre-plane coordinates
    const float fu = div_by(u, du_iso, inv_du) + cu;
    // floor(fu) >= 0 and floor(fu) + 1 < nu (false for a NaN)
    const bool u_in = fu >= 0.f && fu < u_top;
    const float fl = floor_of(fu);
    const int u0 = u_in ? whole(fl) : 0;
    const float au = fraction(fu, fl);
    const float bu = 1.f - au, m2 = mag * mag;
    if constexpr (ZB <= 2) {
      // few warps: every tap is loaded before any is used (a voxel outside the panel reads a word it leaves out)
      float av[ZB], t[ZB][4];
      bool in[ZB];
#pragma unroll
      for (int j = 0; j < ZB; ++j) {
        const float v = z[j] * mag;
        const float fv = div_by(v, dv_iso, inv_dv) + cv;
        const float fw = floor_of(fv);
        av[j] = fraction(fv, fw);
        in[j] = u_in && fv >= 0.f && fv < v_top;
        const float* r0 = in[j] ? row(fw, u0) : q;
        t[j][0] = __ldg(r0);
        t[j][1] = __ldg(r0 + 1);
        t[j][2] = __ldg(r0 + nu);
        t[j][3] = __ldg(r0 + nu + 1);
      }
#pragma unroll
      for (int j = 0; j < ZB; ++j) {
        const float val = (1.f - av[j]) * (bu * t[j][0] + au * t[j][1]) + av[j] * (bu * t[j][2] + au * t[j][3]);
        acc[j] = fmaf(m2, in[j] ? val : 0.f, acc[j]);
      }
    } else {
#pragma unroll
      for (int j = 0; j < ZB; ++j) {
        const float v = z[j] * mag;
        const float fv = div_by(v, dv_iso, inv_dv) + cv;
        const float fw = floor_of(fv);
        const float av = fraction(fv, fw);
        float val = 0.f;
        if (u_in && fv >= 0.f && fv < v_top) {
          const float* r0 = row(fw, u0);
          const float* r1 = r0 + nu;
          val = (1.f - av) * (bu * __ldg(r0) + au * __ldg(r0 + 1)) + av * (bu * __ldg(r1) + au * __ldg(r1 + 1));
        }
        acc[j] = fmaf(m2, val, acc[j]);
      }
    }
  }
#pragma unroll
  for (int j = 0; j < ZB; ++j)
    if (iz0 + j < nz) vol[((size_t)(iz0 + j) * ny + iy) * nx + ix] = acc[j] * scale;
}

template <int ZB>
cudaError_t backproject(const float* q, const float* cb, const float* sb, int n_proj, int nu, int nv, float du, float dv,
                        float sod, int nx, int ny, int nz, float dx, float dy, float dz, bool first,
                        float scale, float* vol, cudaStream_t s) {
  const long long blocks = (long long)((nx + 15) / 16) * ((ny + 15) / 16) * ((nz + ZB - 1) / ZB);
  if (blocks > 0x7FFFFFFFll) return cudaErrorInvalidValue;
  auto* k = (size_t)nu * nv > 0x7FFFFFFFu || nv > 1 << 22 ? k_fdk_backproject<ZB, true> : k_fdk_backproject<ZB, false>;
  k<<<(unsigned)blocks, 256, 0, s>>>(q, cb, sb, n_proj, nu, nv, du, dv, 1.f / du, 1.f / dv, sod, nx, ny, nz, dx, dy, dz,
                                     first ? 1 : 0, scale, vol);
  return cudaGetLastError();
}

// Rows longer than the transforms of k_ramp.cu take.
cudaError_t filter_direct(const float* p, int nu, int nv, int rows_total, float du, float dv, float sod, float* q,
                          cudaStream_t s) {
  const int span = kFiltThreads * kFiltOut;
  const size_t npad = ((size_t)nu + span - 1) / span * span;
  const size_t smem = ((2 * (npad + kFiltOut) + 1) + (size_t)kFiltRows * nu) * 4;
  if (smem > 200 * 1024) return cudaErrorInvalidValue;
  cudaError_t e = cudaFuncSetAttribute(k_fdk_filter, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  k_fdk_filter<<<(rows_total + kFiltRows - 1) / kFiltRows, kFiltThreads, smem, s>>>(p, nu, nv, rows_total, du, dv, sod,
                                                                                    q);
  return cudaGetLastError();
}

constexpr int kBins = 256;

__device__ __forceinline__ int bin_of(float v, float lo, float sc) {
  return min(max((int)((v - lo) * sc), 0), kBins - 1);
}

// Histogram of vol over [lo, hi) in kBins bins (values outside are clamped to
// the end bins).  A volume's voxels crowd a few bins (air, water), where one
// shared counter per bin serialises a warp: each lane counts in its own copy
// (copy = lane = bank).  256^3: 39 -> 18 us.
__global__ void __launch_bounds__(256) k_hist(const float* __restrict__ vol, size_t n, float lo, float hi,
                                              unsigned int* __restrict__ hist) {
  __shared__ unsigned int sh[kBins * 32];
  for (int b = threadIdx.x; b < kBins * 32; b += blockDim.x) sh[b] = 0;
  __syncthreads();
  const int lane = threadIdx.x & 31;
  const float sc = (float)kBins / (hi - lo);
  const size_t n4 = ((uintptr_t)vol & 15) == 0 ? n / 4 : 0;
  for (size_t i = gtid(); i < n4; i += gstride()) {
    const float4 v = __ldg(reinterpret_cast<const float4*>(vol) + i);
    atomicAdd(&sh[bin_of(v.x, lo, sc) * 32 + lane], 1u);
    atomicAdd(&sh[bin_of(v.y, lo, sc) * 32 + lane], 1u);
    atomicAdd(&sh[bin_of(v.z, lo, sc) * 32 + lane], 1u);
    atomicAdd(&sh[bin_of(v.w, lo, sc) * 32 + lane], 1u);
  }
  for (size_t i = 4 * n4 + gtid(); i < n; i += gstride()) atomicAdd(&sh[bin_of(vol[i], lo, sc) * 32 + lane], 1u);
  __syncthreads();
  for (int b = threadIdx.x; b < kBins; b += blockDim.x) {
    unsigned int t = 0;
    for (int k = 0; k < 32; ++k) t += sh[b * 32 + ((k + b) & 31)];
    if (t) atomicAdd(&hist[b], t);
  }
}

// Multi-level Otsu (classes = 2 or 3): thresholds maximising the between-class
// variance of the histogram, exhaustively, ties to the smallest.  Bound by the
// FP64 divisions of its 32640 candidates, two lanes a clock and SM: block a - 1
// takes the candidates with first threshold a, thread b - 1 the second threshold
// b, and the last block to finish picks the best (one block over all: 563 us).
struct OtsuScratch {
  double val[kBins];
  int second[kBins];
  unsigned int done;
};
__global__ void __launch_bounds__(kBins) k_otsu(const unsigned int* __restrict__ hist, int classes, OtsuScratch* sc,
                                                int* __restrict__ thr) {
  __shared__ double P[kBins + 1], S[kBins + 1];
  __shared__ double val[kBins];
  __shared__ int at[kBins];
  __shared__ bool last;
  const int t = threadIdx.x;
  // counts and count-weighted bin centres are multiples of 1/2 below 2^52: their sums are exact in any order
  if (t == 0) P[0] = S[0] = 0.0;
  P[t + 1] = (double)hist[t];
  S[t + 1] = (double)hist[t] * (t + 0.5);
  __syncthreads();
  for (int o = 1; o < kBins; o <<= 1) {
    const double p = t >= o ? P[t + 1 - o] : 0.0, s = t >= o ? S[t + 1 - o] : 0.0;
    __syncthreads();
    P[t + 1] += p;
    S[t + 1] += s;
    __syncthreads();
  }
  const double N = P[kBins], mu = S[kBins] / fmax(N, 1.0);
  auto term = [&](int a, int b) {  // class [a, b)
    const double w = P[b] - P[a];
    if (w <= 0) return 0.0;
    const double m = (S[b] - S[a]) / w;
    return w * (m - mu) * (m - mu);
  };
  const int a = 1 + blockIdx.x;  // first threshold, 1 .. kBins - 1
  double v = -1.0;
  int b = kBins;
  if (classes == 2) {
    if (t == 0) v = term(0, a) + term(a, kBins);
  } else {
    const int bb = 1 + t;
    if (bb > a && bb < kBins) {
      v = term(0, a) + term(a, bb) + term(bb, kBins);
      b = bb;
    }
  }
  val[t] = v;
  at[t] = b;
  __syncthreads();
  // largest value, the smallest index among equals
  auto best = [&]() {
    for (int o = kBins / 2; o > 0; o >>= 1) {
      if (t < o && (val[t + o] > val[t] || (val[t + o] == val[t] && at[t + o] < at[t]))) {
        val[t] = val[t + o];
        at[t] = at[t + o];
      }
      __syncthreads();
    }
  };
  best();
  if (t == 0) {
    sc->val[a] = val[0];
    sc->second[a] = at[0];
    __threadfence();
    last = atomicAdd(&sc->done, 1u) == gridDim.x - 1;
  }
  __syncthreads();
  if (!last) return;
  __threadfence();
  val[t] = t >= 1 ? __ldcg(sc->val + t) : -2.0;
  at[t] = t;
  __syncthreads();
  best();
  if (t == 0) {
    // without a candidate (no second threshold above the first): the first pair
    thr[0] = val[0] >= 0.0 ? at[0] : 1;
    thr[1] = val[0] >= 0.0 ? __ldcg(sc->second + at[0]) : kBins;
  }
}

// Class of each voxel by the thresholds (bins) -> material id and density
// rho = mu / (mu_rho(material) * 0.1), clamped to [0, rho_max]; class 0 -> the
// background material at its nominal density.  Four voxels per thread where the
// arrays are aligned for it.
__global__ void __launch_bounds__(256) k_segment(const float* __restrict__ vol, size_t n, float lo, float hi,
                                                 const int* __restrict__ thr, int classes, SegmentClasses cls,
                                                 float rho_max, uint8_t* __restrict__ mat, uint16_t* __restrict__ rho) {
  const float sc = (float)kBins / (hi - lo);
  const int t0 = thr[0], t1 = thr[1];
  auto voxel = [&](float v, uint8_t& m, uint16_t& d) {
    const int b = bin_of(v, lo, sc);
    const int c = b < t0 ? 0 : ((classes == 2 || b < t1) ? 1 : 2);
    m = (uint8_t)(c == 0 ? cls.mat[0] : c == 1 ? cls.mat[1] : cls.mat[2]);
    const float r = c == 0 ? cls.rho0 : fminf(fmaxf(v / (0.1f * (c == 1 ? cls.murho[1] : cls.murho[2])), 0.f), rho_max);
    d = __half_as_ushort(__float2half_rn(r));
  };
  const bool wide = ((uintptr_t)vol & 15) == 0 && ((uintptr_t)mat & 3) == 0 && ((uintptr_t)rho & 7) == 0;
  const size_t n4 = wide ? n / 4 : 0;
  for (size_t i = gtid(); i < n4; i += gstride()) {
    const float4 v = __ldg(reinterpret_cast<const float4*>(vol) + i);
    uchar4 m;
    ushort4 d;
    voxel(v.x, m.x, d.x);
    voxel(v.y, m.y, d.y);
    voxel(v.z, m.z, d.z);
    voxel(v.w, m.w, d.w);
    reinterpret_cast<uchar4*>(mat)[i] = m;
    reinterpret_cast<ushort4*>(rho)[i] = d;
  }
  for (size_t i = 4 * n4 + gtid(); i < n; i += gstride()) voxel(vol[i], mat[i], rho[i]);
}

// Down-sampling by 2 per axis for the Monte Carlo step (Sec. II-C.2, II-E):
// each 2x2x2 block becomes one voxel of the material with the block's largest
// mass (ties to the lower id) and the density that keeps the block's summed
// attenuation at the effective energy, sum_v murho[m_v] rho_v / (8 murho[m_b]).
__global__ void __launch_bounds__(256) k_bin_volume(const uint8_t* __restrict__ mat, const uint16_t* __restrict__ rho,
                                                    int nx, int ny, int nz, MaterialValues murho, int n_mat,
                                                    uint8_t* __restrict__ mat_b, uint16_t* __restrict__ rho_b) {
  const int bx = nx / 2, by = ny / 2, bz = nz / 2;
  const size_t n = (size_t)bx * by * bz;
  __shared__ float s_mu[256];  // for every id a voxel can hold; one in no table attenuates nothing
  for (int m = threadIdx.x; m < 256; m += blockDim.x) s_mu[m] = m < n_mat ? murho.v[m] : 0.f;
  __syncthreads();
  // a block's x neighbours as one 2- and one 4-byte word (nx is even, so rows keep the arrays' alignment)
  const bool wide = ((uintptr_t)mat & 1) == 0 && ((uintptr_t)rho & 3) == 0;
  for (size_t i = gtid(); i < n; i += gstride()) {
    const size_t row = i / bx;
    const int x = (int)(i - row * bx), y = (int)(row % by), z = (int)(row / by);
    float mass[kMaxMat];
#pragma unroll
    for (int m = 0; m < kMaxMat; ++m) mass[m] = 0.f;
    float mu = 0.f;
#pragma unroll
    for (int p = 0; p < 4; ++p) {
      const size_t v = ((size_t)(2 * z + (p >> 1)) * ny + (2 * y + (p & 1))) * nx + 2 * x;
      const uint32_t mm = wide ? __ldg(reinterpret_cast<const uint16_t*>(mat + v)) : mat[v] | ((uint32_t)mat[v + 1] << 8);
      const uint32_t rr = wide ? __ldg(reinterpret_cast<const uint32_t*>(rho + v)) : rho[v] | ((uint32_t)rho[v + 1] << 16);
#pragma unroll
      for (int q = 0; q < 2; ++q) {
        const int m = (mm >> (8 * q)) & 255u;
        const float r = __half2float(__ushort_as_half((unsigned short)(rr >> (16 * q))));
#pragma unroll
        for (int k = 0; k < kMaxMat; ++k) mass[k] += (k == m) ? r : 0.f;
        mu = fmaf(s_mu[m], r, mu);
      }
    }
    int best = 0;
    float top = mass[0];
#pragma unroll
    for (int m = 1; m < kMaxMat; ++m)
      if (m < n_mat && mass[m] > top) {
        top = mass[m];
        best = m;
      }
    mat_b[i] = (uint8_t)best;
    rho_b[i] = __half_as_ushort(__float2half_rn(mu / (8.f * s_mu[best])));
  }
}

// c = a - ln(Ip / (Ip + Is)) (eq. Correction).
__global__ void k_correct(const float* __restrict__ a, const float* __restrict__ ip, const float* __restrict__ is,
                          float is_scale, size_t n, float* __restrict__ c) {
  for (size_t i = gtid(); i < n; i += gstride()) {
    const float p = fmaxf(ip[i], 1e-30f), sc = fmaxf(is[i], 0.f) * is_scale;
    c[i] = a[i] - logf(p / (p + sc));
  }
}

}  // namespace

cudaError_t recon_bin_volume(const uint8_t* mat, const uint16_t* rho, int nx, int ny, int nz,
                             const MaterialValues& murho, int n_mat, uint8_t* mat_b, uint16_t* rho_b, cudaStream_t s) {
  if (nx % 2 || ny % 2 || nz % 2 || n_mat < 1 || n_mat > kMaxMat) return cudaErrorInvalidValue;
  const size_t n = (size_t)(nx / 2) * (ny / 2) * (nz / 2);
  k_bin_volume<<<blocks_for(n), 256, 0, s>>>(mat, rho, nx, ny, nz, murho, n_mat, mat_b, rho_b);
  return cudaGetLastError();
}

cudaError_t recon_log_norm(const float* I, const float* I0, size_t img, size_t n, float* a, cudaStream_t s) {
  k_log_norm<<<blocks_for(n), 256, 0, s>>>(I, I0, img, n, a);
  return cudaGetLastError();
}

cudaError_t recon_fdk(const float* p, int n_proj, const float* d_cos, const float* d_sin, int nu, int nv, float pu,
                      float pv, float sod, float sdd, int nx, int ny, int nz, float dx, float dy, float dz,
                      float* d_ramp, int chunk, float* q_tmp, float* vol, cudaStream_t s) {
  const float du = pu * sod / sdd, dv = pv * sod / sdd;  // pixel pitch at the isocentre
  // full orbit: (dbeta / 2) with dbeta = 2 pi / n_proj
  const float scale = 3.14159265358979f / (float)n_proj;
  const size_t img = (size_t)nu * nv;
  // 8 voxels of a column per thread share its source-side terms; with fewer than about 16 blocks per SM of them, 2
  // (200^3 x 128 projections, 4225 blocks: 1.56 / 1.72 ms with 8 / 2; 128^3 x 360, 1024 blocks: 2.2 / 1.7)
  const bool deep = (long long)((nx + 15) / 16) * ((ny + 15) / 16) * ((nz + 7) / 8) >= 16ll * 152;
  for (int k = 0; k < n_proj; k += chunk) {
    const int m = n_proj - k < chunk ? n_proj - k : chunk;
    cudaError_t e = d_ramp ? ramp_filter(p + k * img, nu, nv, m * nv, du, dv, sod, d_ramp, q_tmp, k == 0, s)
                           : filter_direct(p + k * img, nu, nv, m * nv, du, dv, sod, q_tmp, s);
    if (e != cudaSuccess) return e;
    const float sc = k + m == n_proj ? scale : 1.f;
    e = deep ? backproject<8>(q_tmp, d_cos + k, d_sin + k, m, nu, nv, du, dv, sod, nx, ny, nz, dx, dy, dz, k == 0, sc, vol, s)
             : backproject<2>(q_tmp, d_cos + k, d_sin + k, m, nu, nv, du, dv, sod, nx, ny, nz, dx, dy, dz, k == 0, sc, vol, s);
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

size_t recon_segment_scratch() { return kBins * 4 + 16 + sizeof(OtsuScratch); }

cudaError_t recon_otsu_segment(const float* vol, size_t n, float lo, float hi, int classes, const SegmentClasses& cls,
                               float rho_max, void* scratch, unsigned int** d_hist, int** d_thr, uint8_t* mat,
                               uint16_t* rho, cudaStream_t s) {
  unsigned int* hist = static_cast<unsigned int*>(scratch);
  int* thr = reinterpret_cast<int*>(hist + kBins);
  OtsuScratch* otsu = reinterpret_cast<OtsuScratch*>(thr + 4);
  *d_hist = hist;
  *d_thr = thr;
  cudaError_t e = cudaMemsetAsync(scratch, 0, recon_segment_scratch(), s);
  if (e != cudaSuccess) return e;
  // few blocks: each zeroes and sums 32 copies of the histogram
  const int grid = blocks_for((n + 3) / 4) < 152 * 4 ? blocks_for((n + 3) / 4) : 152 * 4;
  k_hist<<<grid, 256, 0, s>>>(vol, n, lo, hi, hist);
  k_otsu<<<kBins - 1, kBins, 0, s>>>(hist, classes, otsu, thr);
  k_segment<<<blocks_for((n + 3) / 4), 256, 0, s>>>(vol, n, lo, hi, thr, classes, cls, rho_max, mat, rho);
  return cudaGetLastError();
}

cudaError_t recon_correct(const float* a, const float* ip, const float* is, float is_scale, size_t n, float* c,
                          cudaStream_t s) {
  k_correct<<<blocks_for(n), 256, 0, s>>>(a, ip, is, is_scale, n, c);
  return cudaGetLastError();
}

}  // namespace mcx

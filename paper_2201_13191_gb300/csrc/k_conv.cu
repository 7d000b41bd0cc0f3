// 3x3 convolutions of the learned scatter denoiser on the tcgen05 tensor cores.
//
// Tensors are NHWC, BF16, with channel counts that are multiples of 16.
//  - forward: implicit GEMM over shifted views of a halo tile fetched by the
//    tensor memory accelerator (description at k_conv3x3_fwd); FP32
//    accumulators in tensor memory; epilogue bias, optional ReLU, BF16 or FP32.
//  - input gradient: the same kernel with the adjoint weights (flipped in space,
//    transposed in channels: a 3x3 'same' convolution's adjoint).
//  - weight gradient: both operands MN-major from tiled copies, the reduction
//    over pixels (description at k_conv3x3_wgrad); CTAs split the pixels and add
//    their FP32 partial tiles into dW.
#include <cuda.h>
#include <cuda_bf16.h>
#include <stdint.h>

#include <algorithm>
#include <mutex>

#include "mc_internal.h"
#include "mc_tc.cuh"

namespace mcx {
namespace {

constexpr int kThreads = 128;  // four warps: one per 32 tensor-memory lanes

// ---------------------------------------------------------------------------
// Forward (and input-gradient) convolution.
//
// Tiling.  The image is cut into column strips of width ws = min(w, MC_CONV_WS); a
// strip with its one-pixel border (the neighbouring strips' columns, or zeros
// at the image edge) and a zero row above and below is the "padded strip", of
// width wp = ws + 2, linearised row-major.  A CTA computes A x 128 consecutive
// positions q of one padded strip (A accumulators of 128 rows x N output
// channels in tensor memory); positions on the border are computed and
// discarded.  For tap (dy, dx) the input of position q sits at q + dy*wp + dx,
// so with the input tile ("halo": the rows of the padded strip that cover
// [q0 - wp - 1, q0 + 128A + wp]) stored position-major -- one row of CC
// channels (2 CC bytes, swizzled 32/64/128B) per position, the canonical
// K-major swizzled layout -- every tap's A operand is the same tile seen from
// a start address shifted by (dy*wp + dx) rows.  Each input chunk is fetched
// once per CTA instead of nine times, by one tiled 4-D tensor copy per stage
// (zero-filled outside the image).
//
// Pipeline.  The reduction runs over the input channels in chunks of CC; a
// chunk's stage holds its halo and its weights for all nine taps (the packed
// operand order wm[ci/8][tap][co][ci%8] makes that one contiguous block).
// Warp 0 lane 0 fills a ring of `stages` stages (mbarrier `full`), warp 1
// lane 0 issues the MMAs (9 taps x CC/16 k-steps x A accumulators per stage)
// and frees each stage with tcgen05.commit (mbarrier `empty`); after the last
// stage all four warps read their accumulator rows (tensor-memory lanes) and
// store bias + optional ReLU, BF16 or FP32.
// ---------------------------------------------------------------------------
constexpr int kMaxStages = 8;
constexpr int kSmemBudget = 225 * 1024;  // the most one CTA may take
// Shared memory the planner lets one forward CTA take: the whole budget (one
// CTA per SM, the deepest ring) or less, so that several CTAs share an SM and
// one's pipeline fill and epilogue overlap another's MMAs.
#ifndef MC_CONV_PLAN_KB
#define MC_CONV_PLAN_KB 110
#endif
constexpr int kPlanBudget = MC_CONV_PLAN_KB * 1024;
// Output-channel tiles narrower than C_out when the grid would not cover the
// SMs (1), or always C_out rounded up (0).
#ifndef MC_CONV_SPLIT_N
#define MC_CONV_SPLIT_N 1
#endif
// Widest strip (columns) the forward tiles cut an image into: narrower strips
// cut the halo rows a tile fetches (measured 301.6 / 307.9 / 312.3 TFLOP/s
// FLOP-weighted at 128 / 64 / 32 over the denoiser's layers).
#ifndef MC_CONV_WS
#define MC_CONV_WS 32
#endif

struct FwdArgs {
  const __nv_bfloat16* wm;  // packed weights [cin/8][9][co_total][8]
  const float* bias;        // [cout] or null
  void* y;                  // [n][h][w][cout]
  int n, h, w, cin, cout, co_total, co0;
  int ws, strips, wp, tiles;  // strip width, strips per row, padded width, tiles per strip
  int A, CC, stages, rbox;    // accumulators, channels per stage, ring depth, halo rows per copy
  uint32_t halo_bytes, stage_bytes;
  int rb;                     // halo bytes per position row (2 CC), swizzled in 8-row groups
  int relu, out_f32;
  int* err;
};

__device__ __forceinline__ uint32_t tmem_cols(int n) {
  uint32_t c = 32;
  while (c < (uint32_t)n) c <<= 1;
  return c;
}

// Tap folding (FOLD, for C_out tiles with 3N <= 256).  The three taps of one
// kernel row (dy, dx = -1, 0, +1) share one MMA: the A operand is the halo seen
// from the row shift dy*wp - 1 alone and B holds the three taps' weights side by
// side (N_mma = 3N, contiguous in the packed [tap][co] order), so accumulator
// row r collects, in column block dx, the contributions that output position
// r - 1 - dx ... needs; the epilogue adds block -1 of row r, block 0 of row
// r + 1 and block +1 of row r + 2.  That is 3 instead of 9 MMAs per k-step,
// each three times wider (narrow-N MMAs are bound by their A operand reads),
// and 126 instead of 128 output positions per accumulator.
#ifndef MC_CONV_FOLD
#define MC_CONV_FOLD 1
#endif
constexpr int kFoldRows = 126;

template <int N, bool FOLD>
__global__ void __launch_bounds__(kThreads, 1) k_conv3x3_fwd(const __grid_constant__ CUtensorMap xmap, const FwdArgs a) {
  extern __shared__ unsigned char dyn_raw[];
  unsigned char* sm = reinterpret_cast<unsigned char*>(((uintptr_t)dyn_raw + 1023) & ~(uintptr_t)1023);
  __shared__ __align__(8) uint64_t full[kMaxStages], empty[kMaxStages], done;
  __shared__ uint32_t tmem_holder;
  __shared__ volatile int abort_flag;
  const int tid = threadIdx.x, warp = __shfl_sync(0xFFFFFFFFu, tid >> 5, 0), lane = tid & 31;

  int tile = blockIdx.x;
  const int t = tile % a.tiles;
  tile /= a.tiles;
  const int strip = tile % a.strips;
  const int img = tile / a.strips;
  const int nb = blockIdx.y * N;  // first output channel of this CTA (within the launch's cout)
  constexpr int NA = FOLD ? 3 * N : N;         // accumulator columns
  constexpr int RA = FOLD ? kFoldRows : 128;   // output positions per accumulator
  const int Mt = RA * a.A;
  const int q0 = a.wp + 1 + t * Mt;           // first position: row 1, column 1 of the padded strip
  const int vr_lo = (q0 - a.wp - 1) / a.wp;   // first halo row (padded-strip row index)
  const int o0 = q0 - vr_lo * a.wp;           // halo index of q0
  const int n_chunks = a.cin / a.CC;
  const uint32_t ncols = tmem_cols(a.A * NA);

  if (warp == 0) tc::tmem_alloc(&tmem_holder, ncols);
  if (tid == 0) {
    for (int i = 0; i < a.stages; ++i) {
      tc::mbar_init(&full[i], 1);
      tc::mbar_init(&empty[i], 1);
    }
    tc::mbar_init(&done, 1);
    abort_flag = 0;
  }
  tc::fence_before();
  __syncthreads();
  tc::fence_after();
  const uint32_t tmem = tmem_holder;

  if (warp == 0) {
    if (lane == 0) {
      // ---- producer: halo by tensor copies, weights by one bulk copy per chunk
      const int rows = min(N, a.cout - nb);  // weight rows this CTA needs
      const int r0 = a.co0 + nb;
      const bool one_block = rows == N && N == a.co_total;
      const uint32_t w_tx = (uint32_t)(a.CC / 8) * 9u * (uint32_t)rows * 16u;
      const uint32_t halo_tx = (uint32_t)(a.CC / 8) * 16u * (uint32_t)a.wp * (uint32_t)a.rbox;
      int issued = 0;
      for (int st = 0; st < n_chunks; ++st) {
        const int slot = st % a.stages;
        if (st >= a.stages && !tc::mbar_wait(&empty[slot], (uint32_t)((st / a.stages) - 1) & 1u)) {
          abort_flag = 1;
          break;
        }
        if (abort_flag) break;
        unsigned char* hs = sm + (size_t)slot * a.stage_bytes;
        unsigned char* wsm = hs + a.halo_bytes;
        tc::mbar_expect_tx(&full[slot], halo_tx + w_tx);
        const int g0 = st * (a.CC / 8);  // first 8-channel group of the chunk
        tc::tma_load_4d(hs, &xmap, &full[slot], g0 * 8, strip * a.ws - 1, vr_lo - 1, img);
        if (one_block) {
          tc::bulk_load(wsm, a.wm + (size_t)g0 * 9 * a.co_total * 8, w_tx, &full[slot]);
        } else {
          for (int kc = 0; kc < a.CC / 8; ++kc)
            for (int tap = 0; tap < 9; ++tap)
              tc::bulk_load(wsm + (size_t)((kc * 9 + tap) * N) * 16,
                            a.wm + ((size_t)((g0 + kc) * 9 + tap) * a.co_total + r0) * 8, (uint32_t)rows * 16u,
                            &full[slot]);
        }
        ++issued;
      }
      if (abort_flag) {
        // let the copies still in flight land before the CTA can exit
        for (int st = max(0, issued - a.stages); st < issued; ++st)
          tc::mbar_wait(&full[st % a.stages], (uint32_t)(st / a.stages) & 1u);
      }
    }
    __syncwarp();
  } else if (warp == 1) {
    {
      // ---- MMA issuer: the whole warp runs the loop and one lane issues, so that the descriptors stay in
      // uniform registers (against one lane's own loop, 64 -> 64 channels at 16 x 128^2: 46.5 -> 40.9 us,
      // 96 -> 32 at 16 x 256^2: 145 -> 122 us)
      const bool lead = tc::elect_one();
      const uint32_t idesc = tc::idesc_bf16(128, NA);
      const uint32_t lbo_b = 9u * N * 16u;
      constexpr int kGroups = FOLD ? 3 : 9;  // MMAs per k-step and accumulator: kernel rows or taps
      for (int st = 0; st < n_chunks; ++st) {
        const int slot = st % a.stages;
        if (!__all_sync(0xFFFFFFFFu, tc::mbar_wait(&full[slot], (uint32_t)(st / a.stages) & 1u))) {
          abort_flag = 1;
          break;
        }
        tc::fence_after();
        const uint32_t hb = tc::saddr(sm + (size_t)slot * a.stage_bytes);
        const uint32_t wb = hb + a.halo_bytes;
        for (int g = 0; g < kGroups; ++g) {
          // first tap of the group and the row shift of its A operand
          const int tap = FOLD ? 3 * g : g;
          const int shift = FOLD ? (g - 1) * a.wp - 1 : (tap / 3 - 1) * a.wp + (tap % 3 - 1);
          for (int ks = 0; ks < a.CC / 16; ++ks) {
            const uint64_t db = tc::sdesc(wb + (uint32_t)((2 * ks * 9 + tap) * N) * 16u, lbo_b, 128);
            for (int acc = 0; acc < a.A; ++acc) {
              // rows of 2 CC bytes, 8-row groups 8 rb apart; k-step = 32 bytes within the row.  The
              // tensor core applies the swizzle on absolute shared-memory address bits, like the TMA
              // that wrote the tile, so a start shifted by any number of rows needs no phase field.
              const uint32_t sa = hb + (uint32_t)(o0 + RA * acc + shift) * (uint32_t)a.rb + (uint32_t)ks * 32u;
              const uint64_t da = tc::sdesc_swz(sa, 8u * (uint32_t)a.rb, a.rb);
              if (lead) tc::mma_bf16(tmem + (uint32_t)(acc * NA), da, db, idesc, (st | g | ks) ? 1u : 0u);
            }
          }
        }
        if (lead) tc::commit(&empty[slot]);
      }
      if (lead) tc::commit(&done);
    }
    __syncwarp();
  }
  bool ok = tc::mbar_wait(&done, 0);
  tc::fence_after();
  // one decision for the whole CTA: the folded epilogue synchronises its threads
  ok = __syncthreads_and(ok && !abort_flag) != 0;
  if (!ok && tid == 0) atomicOr(a.err, 1);
  if (ok) {
    const uint32_t lane_base = tmem + ((uint32_t)(warp * 32) << 16);
    // exchange rows of the folded epilogue: the ring is idle once `done` has completed
    constexpr int kX = 20;  // floats per row (16 used; 80-byte rows keep float4 reads conflict-free)
    float* xch = reinterpret_cast<float*>(sm);
    for (int acc = 0; acc < a.A; ++acc) {
      const int q = q0 + RA * acc + tid;
      const int vr = q / a.wp, vc = q - vr * a.wp;
      const int y = vr - 1, x = strip * a.ws + vc - 1;
      const bool valid = (!FOLD || tid < kFoldRows) && vr >= 1 && vr <= a.h && vc >= 1 && vc <= a.ws && x < a.w;
      const long long pix = ((long long)img * a.h + y) * a.w + x;
      if (N >= 64 && !a.out_f32) {
        // BF16: 32 channels at a time through shared memory, so that neighbouring lanes store neighbouring
        // 16-byte units, 64 contiguous bytes a position instead of one lane's 16 (64 -> 64 channels at
        // 16 x 128^2: 40.9 -> 37.2 us; 128 -> 128 at 16 x 64^2: 28.9 -> 26.4).  Tiles of 32 channels, with
        // five CTAs to an SM, are faster with one lane's stores (96 -> 32 at 16 x 256^2: 122 against 131 us).
        constexpr int kRow = 80;  // bytes: 64 used, 16-byte accesses of 8 rows in different banks
        unsigned char* rows = sm + warp * 32 * kRow;
        const long long mine = valid ? pix : -1;
#pragma unroll 1
        for (int c0 = 0; c0 < N; c0 += 32) {
          float v[32];
          tc::tmem_ld32(lane_base + (uint32_t)(acc * NA + c0), v);
          const int co = nb + c0, left = a.cout - co;  // a multiple of 16
          if (left <= 0) continue;
#pragma unroll
          for (int j = 0; j < 32; ++j) {
            if (a.bias && j < left) v[j] += __ldg(a.bias + co + j);
            if (a.relu) v[j] = fmaxf(v[j], 0.f);
          }
          __syncwarp();  // the previous 32 channels are read
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            __nv_bfloat162 b[4];
#pragma unroll
            for (int m = 0; m < 4; ++m) b[m] = __floats2bfloat162_rn(v[8 * j + 2 * m], v[8 * j + 2 * m + 1]);
            *reinterpret_cast<uint4*>(rows + lane * kRow + 16 * j) = *reinterpret_cast<uint4*>(b);
          }
          __syncwarp();
#pragma unroll
          for (int m = 0; m < 4; ++m) {
            const int row = 8 * m + (lane >> 2), u = lane & 3;
            const long long px = __shfl_sync(0xFFFFFFFFu, mine, row);
            if (px >= 0 && 8 * u < left)
              *reinterpret_cast<uint4*>(reinterpret_cast<__nv_bfloat16*>(a.y) + px * a.cout + co + 8 * u) =
                  *reinterpret_cast<const uint4*>(rows + row * kRow + 16 * u);
          }
        }
        continue;
      }
#pragma unroll 1
      for (int c0 = 0; c0 < N; c0 += 8) {
        float v[8];
        tc::tmem_ld8(lane_base + (uint32_t)(acc * NA + c0), v);
        if (FOLD) {
          float v0[8], vp[8];
          tc::tmem_ld8(lane_base + (uint32_t)(acc * NA + N + c0), v0);
          tc::tmem_ld8(lane_base + (uint32_t)(acc * NA + 2 * N + c0), vp);
          __syncthreads();  // the previous chunk's reads of xch are done
          float4* mine = reinterpret_cast<float4*>(xch + tid * kX);
          mine[0] = make_float4(v0[0], v0[1], v0[2], v0[3]);
          mine[1] = make_float4(v0[4], v0[5], v0[6], v0[7]);
          mine[2] = make_float4(vp[0], vp[1], vp[2], vp[3]);
          mine[3] = make_float4(vp[4], vp[5], vp[6], vp[7]);
          __syncthreads();
          if (tid < kFoldRows) {
            const float4* r1 = reinterpret_cast<const float4*>(xch + (tid + 1) * kX);
            const float4* r2 = reinterpret_cast<const float4*>(xch + (tid + 2) * kX);
            const float4 a0 = r1[0], a1 = r1[1], b0 = r2[2], b1 = r2[3];
            v[0] += a0.x + b0.x; v[1] += a0.y + b0.y; v[2] += a0.z + b0.z; v[3] += a0.w + b0.w;
            v[4] += a1.x + b1.x; v[5] += a1.y + b1.y; v[6] += a1.z + b1.z; v[7] += a1.w + b1.w;
          }
        }
        const int co = nb + c0;
        if (valid && co < a.cout) {
#pragma unroll
          for (int j = 0; j < 8; ++j) {
            if (a.bias) v[j] += __ldg(a.bias + co + j);
            if (a.relu) v[j] = fmaxf(v[j], 0.f);
          }
          if (a.out_f32) {
            float* dst = reinterpret_cast<float*>(a.y) + pix * a.cout + co;
            *reinterpret_cast<float4*>(dst) = make_float4(v[0], v[1], v[2], v[3]);
            *reinterpret_cast<float4*>(dst + 4) = make_float4(v[4], v[5], v[6], v[7]);
          } else {
            __nv_bfloat162 b[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) b[j] = __floats2bfloat162_rn(v[2 * j], v[2 * j + 1]);
            *reinterpret_cast<uint4*>(reinterpret_cast<__nv_bfloat16*>(a.y) + pix * a.cout + co) =
                *reinterpret_cast<uint4*>(b);
          }
        }
      }
    }
  }
  tc::fence_before();
  __syncthreads();
  if (warp == 0) tc::tmem_free(tmem, ncols);
}

// ---------------------------------------------------------------------------
// Weight gradient dW[co][dy, dx][c] = sum_p X(y, x + dx)[c] dY(y - dy, x)[co].
//
// A tensor-core GEMM with the reduction over pixels p = (y, x).  Both tensors
// are channel-minor, so both operands are MN-major.  A stage is a tile of 128
// pixels (32 x 4, or 16 x 8 and 8 x 16 for narrow images) of X with one more
// column on either side (rows of CC channels) and of dY with one more row above
// and below (rows of NT channels), each fetched by one tiled copy (zero-filled
// outside the image) in the canonical swizzled layout.  One MMA takes 16 pixels
// (K) and all nine taps: its M rows are 128 / CC blocks of CC channels, X seen
// from starts one pixel apart (the leading-dimension offset), i.e. dx = -1, 0, +1
// (two MMAs at CC = 64; blocks past dx = +1 fall on rows nobody reads), and its
// 3 NT columns are dY seen from starts one row apart, dy = +1, 0, -1.  Shared
// memory is read once per 9 taps instead of three times with the rows' taps in
// separate MMAs of NT columns (the 15 layers of one step: 1030 -> 690 us), and neither
// operand passes through registers.  In the image's first and last row the MMA
// leaves out the columns of the dy that falls outside, so that a value that is
// not finite meets the same products as in the sum above.  Where the width is no
// multiple of 16 such a value also meets the zeros beside the image (in the last
// column's dx = -1; in 8-wide tiles in the first or last row's third dy): the
// accumulators that this has spoilt are summed again from global memory.
//
// CTA (cin chunk, cout tile, split): the split's tiles, a run of neighbours (its
// partial sums then grow, and round, like those of a run of pixels), go through a
// ring of stages (warp 0 lane 0 copies, warp 1 lane 0 issues the MMAs); at the end
// the four warps add the accumulators into dW (FP32 atomics).  Bound by the tensor
// core's operand reads from shared memory and, at the deep layers, the atomics.
// Measured over the denoiser's layers, 16 images of 256^2: 2.83 -> 0.70 ms per
// step against threads that transposed both operands through registers.
// ---------------------------------------------------------------------------
constexpr int kWgPix = 128;      // pixels of a stage's tile
constexpr int kWgXRows = 160;    // X pixels: 34 x 4, 18 x 8 or 10 x 16
constexpr int kWgYRows = 192;    // dY pixels: 32 x 6, 16 x 10 or 8 x 18
constexpr int kWgMaxStages = 8;

template <int CC, int NT>
struct WgPlan {
  static constexpr int groups = CC == 64 ? 2 : 1;  // MMAs per 16 pixels
  static constexpr int cols = 3 * NT * groups;     // accumulator columns
  static constexpr int ra = 2 * CC, rb = 2 * NT;   // bytes per pixel row
  // X rows, and what the blocks past dx = +1 read after the tile's last
  static constexpr int x_bytes = ((kWgXRows + 8) * ra + 1023) & ~1023;
  static constexpr int dy_bytes = (kWgYRows * rb + 1023) & ~1023;
  static constexpr int stage = x_bytes + dy_bytes;
  // one CTA per SM where the accumulators take more than half of tensor memory
  static constexpr int fit = ((cols > 256 ? 220 : 110) * 1024 - 1024) / stage;
  static constexpr int stages = fit > kWgMaxStages ? kWgMaxStages : fit;
  static constexpr int smem = stages * stage + 1024;
};

struct WgArgs {
  float* dw;
  const __nv_bfloat16 *x, *dy;
  int n, h, w, cin, cout, tx, ty, tiles_x, tiles_y;  // tx x ty: the tile
  int* err;
};

// dW[co .. co + 7][tap_y, tap_x][c] over `count` tiles from `first` on, the products inside the image only.
__device__ __forceinline__ void wgrad_direct(const WgArgs& p, long long first, int count, int c, int co, int tap_y,
                                             int tap_x, float (&sum)[8]) {
  const int per_img = p.tiles_x * p.tiles_y;
#pragma unroll
  for (int i = 0; i < 8; ++i) sum[i] = 0.f;
  for (long long t = first; t < first + count; ++t) {
    const long long img = t / per_img;
    const int r = (int)(t - img * per_img), y0 = (r / p.tiles_x) * p.ty, x0 = (r % p.tiles_x) * p.tx;
    const int xa = max(x0, 1 - tap_x), xb = min(min(x0 + p.tx, p.w), p.w + 1 - tap_x);
    for (int y = max(y0, tap_y - 1); y < min(min(y0 + p.ty, p.h), p.h + tap_y - 1); ++y) {
      const __nv_bfloat16* row_x = p.x + ((img * p.h + y) * p.w + (tap_x - 1)) * p.cin + c;
      const __nv_bfloat16* row_g = p.dy + (img * p.h + y - (tap_y - 1)) * p.w * p.cout + co;
#pragma unroll 4
      for (int x = xa; x < xb; ++x) {
        const float v = __bfloat162float(row_x[(long long)x * p.cin]);
        const uint4 q = __ldg(reinterpret_cast<const uint4*>(row_g + (long long)x * p.cout));
        const uint32_t g[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
        for (int i = 0; i < 8; ++i)
          sum[i] = fmaf(v, __uint_as_float(i & 1 ? g[i >> 1] & 0xFFFF0000u : g[i >> 1] << 16), sum[i]);
      }
      bool nan = true;  // all of them: they stay no numbers
#pragma unroll
      for (int i = 0; i < 8; ++i) nan &= sum[i] != sum[i];
      if (nan) return;
    }
  }
}

// Whether channel c holds a value that is not finite in the last column of `count` tiles from `first` on.
__device__ __forceinline__ bool wgrad_last_column(const WgArgs& p, long long first, int count, int c) {
  const int per_img = p.tiles_x * p.tiles_y;
  float z = 0.f;
  for (long long t = first; t < first + count; ++t) {
    const long long img = t / per_img;
    const int r = (int)(t - img * per_img), y0 = (r / p.tiles_x) * p.ty;
    if (r % p.tiles_x != p.tiles_x - 1) continue;
#pragma unroll 4
    for (int y = y0; y < min(y0 + p.ty, p.h); ++y)
      z = fmaf(__bfloat162float(p.x[((img * p.h + y) * p.w + p.w - 1) * p.cin + c]), 0.f, z);
  }
  return z != 0.f;
}

// RAGGED: the width is no multiple of 16 (a variant of its own: the sums from global memory double the registers).
template <int CC, int NT, bool RAGGED>
__global__ void __launch_bounds__(kThreads) k_conv3x3_wgrad(const __grid_constant__ CUtensorMap xmap,
                                                            const __grid_constant__ CUtensorMap ymap, const WgArgs p) {
  using P = WgPlan<CC, NT>;
  extern __shared__ unsigned char dyn_raw[];
  unsigned char* sm = reinterpret_cast<unsigned char*>(((uintptr_t)dyn_raw + 1023) & ~(uintptr_t)1023);
  __shared__ __align__(8) uint64_t full[P::stages], empty[P::stages], done;
  __shared__ uint32_t tmem_holder;
  __shared__ volatile int abort_flag;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int c0 = blockIdx.x * CC, n0 = blockIdx.y * NT;
  const int per_img = p.tiles_x * p.tiles_y;
  const long long tiles = (long long)p.n * per_img;
  const long long first = tiles * blockIdx.z / gridDim.z;  // this CTA's tiles: a run of them
  const int count = (int)(tiles * (blockIdx.z + 1) / gridDim.z - first);
  const uint32_t ncols = tmem_cols(P::cols);
  if (warp == 0) tc::tmem_alloc(&tmem_holder, ncols);
  if (tid == 0) {
    for (int i = 0; i < P::stages; ++i) {
      tc::mbar_init(&full[i], 1);
      tc::mbar_init(&empty[i], 1);
    }
    tc::mbar_init(&done, 1);
    abort_flag = 0;
  }
  tc::fence_before();
  __syncthreads();
  tc::fence_after();
  const uint32_t tmem = tmem_holder;
  const uint32_t lane_base = tmem + ((uint32_t)(warp * 32) << 16);
  for (int j = 0; j < P::cols; j += 8) tc::tmem_zero8(lane_base + (uint32_t)j);
  tc::tmem_wait_st();
  tc::fence_before();
  __syncthreads();
  tc::fence_after();

  if (warp == 0 && lane == 0) {
    // ---- producer
    const uint32_t bytes = (uint32_t)((p.tx + 2) * p.ty * P::ra + p.tx * (p.ty + 2) * P::rb);
    int issued = 0;
    for (int st = 0; st < count; ++st) {
      const int slot = st % P::stages;
      if (st >= P::stages && !tc::mbar_wait(&empty[slot], (uint32_t)((st / P::stages) - 1) & 1u)) {
        abort_flag = 1;
        break;
      }
      if (abort_flag) break;
      const long long t = first + st;
      const int img = (int)(t / per_img), r = (int)(t - (long long)img * per_img);
      const int y0 = (r / p.tiles_x) * p.ty, x0 = (r % p.tiles_x) * p.tx;
      unsigned char* xs = sm + slot * P::stage;
      tc::mbar_expect_tx(&full[slot], bytes);
      tc::tma_load_4d(xs, &xmap, &full[slot], c0, x0 - 1, y0, img);
      tc::tma_load_4d(xs + P::x_bytes, &ymap, &full[slot], n0, x0, y0 - 1, img);
      ++issued;
    }
    if (abort_flag)  // let the copies still in flight land before the CTA can exit
      for (int st = max(0, issued - P::stages); st < issued; ++st)
        tc::mbar_wait(&full[st % P::stages], (uint32_t)(st / P::stages) & 1u);
  } else if (warp == 1 && lane == 0) {
    // ---- MMA issuer; operands MN-major (instruction descriptor bits 15 and 16)
    constexpr uint32_t mn = (1u << 15) | (1u << 16);
    // the MMA's second 8 pixels of X: the next ones, or the next row's of an 8-wide tile
    const uint32_t next8 = (uint32_t)((p.tx == 8 ? 10 : 8) * P::ra), pitch = (uint32_t)(p.tx * P::rb);
    for (int st = 0; st < count; ++st) {
      const int slot = st % P::stages;
      if (!tc::mbar_wait(&full[slot], (uint32_t)(st / P::stages) & 1u)) {
        abort_flag = 1;
        break;
      }
      tc::fence_after();
      const int r = (int)((first + st) % per_img);
      const int y0 = (r / p.tiles_x) * p.ty, wx = p.w - (r % p.tiles_x) * p.tx;
      const uint32_t xa = tc::saddr(sm + slot * P::stage), ya = xa + P::x_bytes;
      for (int i = 0; i < kWgPix / 16; ++i) {
        const int ky = (i * 16) / p.tx, kx = (i * 16) % p.tx, y = y0 + ky;
        if (y >= p.h || kx >= wx) continue;  // outside the image
        // column blocks j = 0, 1, 2 read dY at row y - 1 + j (an 8-wide tile's MMA has row y + 1 as well)
        const int j0 = y == 0 && p.tx != 8 ? 1 : 0, j1 = y == p.h - 1 ? 2 : 3;
        const uint32_t idesc = tc::idesc_bf16(128, (j1 - j0) * NT) | mn;
        const uint64_t db = tc::sdesc_mn(ya + (uint32_t)(i * 16 * P::rb) + (uint32_t)j0 * pitch, pitch, 8u * P::rb, P::rb);
#pragma unroll
        for (int g = 0; g < P::groups; ++g) {
          // 128 / CC blocks one pixel apart, from dx = -1 (or +1, the second group) on
          const uint64_t da = tc::sdesc_mn(xa + (uint32_t)((ky * (p.tx + 2) + kx + 2 * g) * P::ra), P::ra, next8, P::ra);
          tc::mma_bf16(tmem + (uint32_t)((g * 3 + j0) * NT), da, db, idesc, 1u);
        }
      }
      tc::commit(&empty[slot]);
    }
    tc::commit(&done);
  }
  __syncwarp();
  bool ok = tc::mbar_wait(&done, 0);
  tc::fence_after();
  ok = __syncthreads_and(ok && !abort_flag) != 0;
  if (!ok && tid == 0) atomicOr(p.err, 1);
  if (ok && count > 0) {
    // accumulator row = block of CC channels (dx) x channel
    const int m = warp * 32 + lane, c = m % CC, blk = m / CC;
    auto tap = [&](int a) { return 3 * (2 - a % 3) + blk + 2 * (a / 3); };  // of accumulator a, where blk + 2 (a / 3) < 3
    bool again = false;
    if constexpr (RAGGED) {
      // a pass of its own: with the test inside the loop of the adds the 64 x 64 form takes 44 us instead of 39 (mean of the 208^2 layers)
      constexpr int step = NT >= 32 ? 32 : 8;
#pragma unroll 1
      for (int j0 = 0; j0 < P::cols; j0 += step) {
        float v[step], z = 0.f;  // z: no number if one of v is not finite
        if constexpr (step == 32) tc::tmem_ld32(lane_base + (uint32_t)j0, v);
        else tc::tmem_ld8(lane_base + (uint32_t)j0, v);
#pragma unroll
        for (int j = 0; j < step; j += 4) z += fmaf(v[j], 0.f, v[j + 1] * 0.f) + fmaf(v[j + 2], 0.f, v[j + 3] * 0.f);
        again |= blk + 2 * (j0 / (3 * NT)) < 3 && z != 0.f;
      }
      again = __any_sync(0xFFFFFFFFu, again);
    }
    if (RAGGED && again) {
      // zeros beside the image have met the last column's values in the dx = -1 taps, and in 8-wide tiles values of the
      // first and last row in a third dy
      const bool edge = p.tx == 8 || wgrad_last_column(p, first, count, c0 + c);
#pragma unroll 1
      for (int j = 0; j < P::cols; j += 8) {
        float v[8];
        __syncwarp();
        tc::tmem_ld8(lane_base + (uint32_t)j, v);
        const int a = j / NT, n = n0 + j % NT;
        if (blk + 2 * (a / 3) >= 3) continue;
        bool finite = true;
#pragma unroll
        for (int i = 0; i < 8; ++i) finite &= fabsf(v[i]) < INFINITY;
        if (!finite && edge && (p.tx == 8 || tap(a) % 3 == 0)) {
          float o[8];
          wgrad_direct(p, first, count, c0 + c, n, tap(a) / 3, tap(a) % 3, o);
#pragma unroll
          for (int i = 0; i < 8; ++i) v[i] = fabsf(v[i]) < INFINITY ? v[i] : o[i];
        }
#pragma unroll
        for (int i = 0; i < 8; ++i) atomicAdd(p.dw + ((size_t)(n + i) * 9 + tap(a)) * p.cin + c0 + c, v[i]);
      }
    } else {
#pragma unroll 1
      for (int a = 0; a < 3 * P::groups; ++a) {
        const bool use = blk + 2 * (a / 3) < 3;
        float* dst = p.dw + (size_t)n0 * 9 * p.cin + (size_t)tap(a) * p.cin + c0 + c;
#pragma unroll 1
        for (int j0 = 0; j0 < NT; j0 += 8) {
          float v[8];
          tc::tmem_ld8(lane_base + (uint32_t)(a * NT + j0), v);
          if (use)
#pragma unroll
            for (int j = 0; j < 8; ++j) atomicAdd(dst + (size_t)(j0 + j) * 9 * p.cin, v[j]);
        }
      }
    }
  }
  tc::fence_before();
  __syncthreads();
  if (warp == 0) tc::tmem_free(tmem, ncols);
}

// cuTensorMapEncodeTiled through the runtime's driver entry point (no link
// against the driver library).
using EncodeTiledFn = CUresult (*)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                   const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                   CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeTiledFn encode_tiled() {
  static EncodeTiledFn fn = nullptr;
  static std::once_flag once;
  std::call_once(once, [] {
    void* f = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &f, 12000, cudaEnableDefault, &q) == cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<EncodeTiledFn>(f);
  });
  return fn;
}

// Tiling of one launch.  For each accumulator count A (A x N tensor-memory
// columns <= 512): the channel chunk CC and ring depth that fit shared memory
// (prefer >= 3 stages or every chunk resident, then larger chunks); then the A
// with the smallest estimated time, waves x (positions per CTA + halo rows +
// a fixed per-CTA cost), waves counted with the CTAs that fit on one SM.
// Shared memory of one stage's halo: swizzled rows of 2 CC bytes per position,
// one 1024-byte-aligned region.
uint32_t halo_bytes_for(int CC, int rbox, int wp) {
  return ((uint32_t)rbox * (uint32_t)wp * (uint32_t)(2 * CC) + 1023u) & ~1023u;
}

bool plan_fwd_budget(const ConvParams& p, int N, bool fold, int sms, int budget, FwdArgs& a, int& grid_x,
                     int& grid_y, int& smem);

// The plan within the planning budget, or within the whole budget when no tile fits the smaller one.
bool plan_fwd(const ConvParams& p, int N, bool fold, int sms, FwdArgs& a, int& grid_x, int& grid_y, int& smem) {
  return plan_fwd_budget(p, N, fold, sms, kPlanBudget, a, grid_x, grid_y, smem) ||
         plan_fwd_budget(p, N, fold, sms, kSmemBudget, a, grid_x, grid_y, smem);
}

int tmem_cols_host(int n) {
  int c = 32;
  while (c < n) c <<= 1;
  return c;
}

bool plan_fwd_budget(const ConvParams& p, int N, bool fold, int sms, int budget, FwdArgs& a, int& grid_x,
                     int& grid_y, int& smem) {
  a.ws = p.w < MC_CONV_WS ? p.w : MC_CONV_WS;
  a.strips = (p.w + a.ws - 1) / a.ws;
  a.wp = a.ws + 2;
  grid_y = (p.cout + N - 1) / N;
  const int NA = fold ? 3 * N : N;             // accumulator columns
  const int RA = fold ? kFoldRows : 128;       // output positions per accumulator
  const int min_bytes = 128 * 20 * 4 + 1024;   // the folded epilogue's exchange rows
  double best_cost = -1.0;
  for (int A = 8; A >= 1; A >>= 1) {
    if (A * NA > 512) continue;
    const int Mt = RA * A;
    const int rbox = (Mt + 2 * a.wp + 1) / a.wp + 2;
    if (rbox > 256) continue;
    const int tiles = ((p.h - 1) * a.wp + a.ws + Mt - 1) / Mt;
    const long long grid = (long long)p.n * a.strips * tiles * grid_y;
    if (grid / grid_y > 0x7FFFFFFF) continue;
    int bestCC = 0, bestStages = 0, bestScore = -1;
    uint32_t bestStage = 0;
    for (int CC = 64; CC >= 16; CC >>= 1) {
      if (p.cin % CC) continue;
      const uint32_t halo = halo_bytes_for(CC, rbox, a.wp);
      const uint32_t stage = ((halo + (uint32_t)CC * 9u * N * 2u) + 1023u) & ~1023u;
      const int chunks = p.cin / CC;
      int stages = (int)((budget - 1024) / stage);
      if (stages > kMaxStages) stages = kMaxStages;
      if (stages > chunks) stages = chunks;
      if (stages < 1 || (stages < 2 && chunks > 1)) continue;
      const int score = (stages >= 3 || stages == chunks ? 100 : 0) + CC;
      if (score > bestScore) {
        bestScore = score;
        bestCC = CC;
        bestStages = stages;
        bestStage = stage;
      }
    }
    if (bestScore < 0) continue;
    int bytes = (int)(bestStage * bestStages) + 1024;
    if (fold && bytes < min_bytes) bytes = min_bytes;
    int per_sm = (228 * 1024) / (bytes + 1024);
    const int by_tmem = 512 / tmem_cols_host(A * NA);
    if (per_sm > by_tmem) per_sm = by_tmem;
    if (per_sm < 1) per_sm = 1;
    const long long slots = (long long)sms * per_sm;
    const double waves = (double)((grid + slots - 1) / slots);
    const double cost = waves * (Mt + 2.0 * a.wp + 256.0);
    if (best_cost < 0 || cost < best_cost) {
      best_cost = cost;
      a.A = A;
      a.CC = bestCC;
      a.stages = bestStages;
      a.rbox = rbox;
      a.tiles = tiles;
      a.halo_bytes = halo_bytes_for(bestCC, rbox, a.wp);
      a.rb = 2 * bestCC;
      a.stage_bytes = bestStage;
      grid_x = (int)(grid / grid_y);
      smem = bytes;
    }
  }
  return best_cost >= 0;
}

template <int N, bool FOLD>
cudaError_t launch_fwd_kernel(const CUtensorMap& map, const FwdArgs& a, int gx, int gy, int smem, cudaStream_t s) {
  static unsigned long long smem_set = 0;  // devices on which the attribute was raised
  int dev = 0;
  cudaGetDevice(&dev);
  const unsigned long long bit = 1ull << (dev & 63);
  if (!(smem_set & bit)) {
    const cudaError_t e =
        cudaFuncSetAttribute(k_conv3x3_fwd<N, FOLD>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemBudget + 1024);
    if (e != cudaSuccess) return e;
    smem_set |= bit;
  }
  k_conv3x3_fwd<N, FOLD><<<dim3((unsigned)gx, (unsigned)gy), kThreads, smem, s>>>(map, a);
  return cudaGetLastError();
}

template <int N>
cudaError_t launch_fwd_n(const ConvParams& p, cudaStream_t s) {
  int dev0 = 0, sms = 0;
  cudaGetDevice(&dev0);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev0);
  if (sms < 1) sms = 1;
  constexpr bool fold = MC_CONV_FOLD && N == 16;  // measured: a gain at N = 16 only
  FwdArgs a{};
  int gx = 0, gy = 0, smem = 0;
  if (!plan_fwd(p, N, fold, sms, a, gx, gy, smem)) return cudaErrorInvalidValue;
  a.wm = p.wt;
  a.bias = p.bias;
  a.y = p.y;
  a.n = p.n;
  a.h = p.h;
  a.w = p.w;
  a.cin = p.cin;
  a.cout = p.cout;
  a.co_total = p.co_total;
  a.co0 = p.co0;
  a.relu = p.relu;
  a.out_f32 = p.out_f32;
  a.err = p.err;
  EncodeTiledFn enc = encode_tiled();
  if (!enc) return cudaErrorNotSupported;
  CUtensorMap map;
  const cuuint64_t dims[4] = {(cuuint64_t)p.cin, (cuuint64_t)p.w, (cuuint64_t)p.h, (cuuint64_t)p.n};
  const cuuint64_t strides[3] = {(cuuint64_t)p.cin * 2, (cuuint64_t)p.cin * 2 * p.w, (cuuint64_t)p.cin * 2 * p.w * p.h};
  const cuuint32_t box[4] = {(cuuint32_t)a.CC, (cuuint32_t)a.wp, (cuuint32_t)a.rbox, 1u};
  const cuuint32_t estr[4] = {1u, 1u, 1u, 1u};
  const CUtensorMapSwizzle swz = a.rb == 128 ? CU_TENSOR_MAP_SWIZZLE_128B
                                 : a.rb == 64 ? CU_TENSOR_MAP_SWIZZLE_64B
                                              : CU_TENSOR_MAP_SWIZZLE_32B;
  if (enc(&map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, (void*)p.x, dims, strides, box, estr,
          CU_TENSOR_MAP_INTERLEAVE_NONE, swz, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
          CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
    return cudaErrorInvalidValue;
  if constexpr (fold)
    return launch_fwd_kernel<N, true>(map, a, gx, gy, smem, s);
  else
    return launch_fwd_kernel<N, false>(map, a, gx, gy, smem, s);
}

CUtensorMapSwizzle swizzle_of(int row_bytes) {
  return row_bytes == 128 ? CU_TENSOR_MAP_SWIZZLE_128B
                          : row_bytes == 64 ? CU_TENSOR_MAP_SWIZZLE_64B : CU_TENSOR_MAP_SWIZZLE_32B;
}

// Map of an NHWC BF16 tensor with boxes of `ch` channels x bw x bh pixels of one image.
bool nhwc_map(EncodeTiledFn enc, CUtensorMap* map, const void* x, int n, int h, int w, int c, int ch, int bw, int bh) {
  const cuuint64_t dims[4] = {(cuuint64_t)c, (cuuint64_t)w, (cuuint64_t)h, (cuuint64_t)n};
  const cuuint64_t strides[3] = {(cuuint64_t)c * 2, (cuuint64_t)c * 2 * w, (cuuint64_t)c * 2 * w * h};
  const cuuint32_t box[4] = {(cuuint32_t)ch, (cuuint32_t)bw, (cuuint32_t)bh, 1u};
  const cuuint32_t estr[4] = {1u, 1u, 1u, 1u};
  return enc(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, (void*)x, dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
             swizzle_of(2 * ch), CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

int wgrad_tile(int w) { return w > 16 ? 32 : w > 8 ? 16 : 8; }

template <int CC, int NT>
cudaError_t launch_wgrad_n(const WgradParams& p, int splits, cudaStream_t s) {
  using P = WgPlan<CC, NT>;
  EncodeTiledFn enc = encode_tiled();
  if (!enc) return cudaErrorNotSupported;
  WgArgs a;
  a.tx = wgrad_tile(p.w);
  a.ty = kWgPix / a.tx;
  CUtensorMap xmap, ymap;
  if (!nhwc_map(enc, &xmap, p.x, p.n, p.h, p.w, p.cin, CC, a.tx + 2, a.ty) ||
      !nhwc_map(enc, &ymap, p.dy, p.n, p.h, p.w, p.cout, NT, a.tx, a.ty + 2))
    return cudaErrorInvalidValue;
  auto* k = p.w % 16 ? k_conv3x3_wgrad<CC, NT, true> : k_conv3x3_wgrad<CC, NT, false>;
  cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, P::smem);
  if (e != cudaSuccess) return e;
  a.dw = p.dw;
  a.x = p.x;
  a.dy = p.dy;
  a.n = p.n;
  a.h = p.h;
  a.w = p.w;
  a.cin = p.cin;
  a.cout = p.cout;
  a.tiles_x = (p.w + a.tx - 1) / a.tx;
  a.tiles_y = (p.h + a.ty - 1) / a.ty;
  a.err = p.err;
  k<<<dim3(p.cin / CC, p.cout / NT, splits), kThreads, P::smem, s>>>(xmap, ymap, a);
  return cudaGetLastError();
}

template <int CC>
cudaError_t launch_wgrad_c(const WgradParams& p, int splits, cudaStream_t s) {
  if (p.cout % 64 == 0) return launch_wgrad_n<CC, 64>(p, splits, s);
  if (p.cout % 32 == 0) return launch_wgrad_n<CC, 32>(p, splits, s);
  return launch_wgrad_n<CC, 16>(p, splits, s);
}

}  // namespace

// N = the launch's cout rounded up to the tile widths 16/32/64/128/256 (cout a
// multiple of 16; wider outputs are split over blockIdx.y).  x must be 16-byte
// aligned; wt is the packed operand order [cin/8][9][co_total][8].
cudaError_t launch_conv3x3_fwd(const ConvParams& p, cudaStream_t s) {
  if (p.cin % 16 || p.cout % 16 || p.cin < 16 || p.cout < 16 || p.co_total < p.co0 + p.cout || p.n < 1 || p.h < 1 ||
      p.w < 1 || ((uintptr_t)p.x & 15) || ((uintptr_t)p.wt & 15))
    return cudaErrorInvalidValue;
  int N = p.cout <= 16 ? 16 : p.cout <= 32 ? 32 : p.cout <= 64 ? 64 : p.cout <= 128 ? 128 : 256;
  if (MC_CONV_SPLIT_N) {
    // small images: narrower output-channel tiles (more CTAs, each reading the same input tile) until the
    // grid covers the SMs
    int dev = 0, sms = 1;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    while (N > 64) {
      FwdArgs a{};
      int gx = 0, gy = 0, smem = 0;
      if (!plan_fwd(p, N, false, sms, a, gx, gy, smem) || (long long)gx * gy >= sms) break;
      N >>= 1;
    }
  }
  switch (N) {
    case 16: return launch_fwd_n<16>(p, s);
    case 32: return launch_fwd_n<32>(p, s);
    case 64: return launch_fwd_n<64>(p, s);
    case 128: return launch_fwd_n<128>(p, s);
    default: return launch_fwd_n<256>(p, s);
  }
}

// Channel chunks of 64, 32 or 16 (whichever divides the count); x and dy 16-byte aligned.
cudaError_t launch_conv3x3_wgrad(const WgradParams& p, int splits, cudaStream_t s) {
  if (p.cin % 16 || p.cout % 16 || p.cout > 256 || p.cin < 16 || p.cout < 16 || splits < 1 || splits > 65535 ||
      ((uintptr_t)p.x & 15) || ((uintptr_t)p.dy & 15))
    return cudaErrorInvalidValue;
  if (p.cin % 64 == 0) return launch_wgrad_c<64>(p, splits, s);
  if (p.cin % 32 == 0) return launch_wgrad_c<32>(p, splits, s);
  return launch_wgrad_c<16>(p, splits, s);
}

// CTAs that share the pixels: 608 per 128 rows of (tap, channel), each with 256
// pixels at least, rounded up to whole waves (one CTA per SM where its
// accumulators take more than half of tensor memory, else two).  The first sets
// the length of an FP32 sum and so its error, which grows with it (32 -> 32
// channels at 16 x 256^2 against FP64: 7.6e-6, 3.7e-6 and 1.8e-6 of the norm with
// 152, 304 and 608 CTAs).  Whole waves: 32 -> 32, 203 CTAs 48 us, 304 37; 64 -> 64
// at 128^2, 122 CTAs 40 us, 152 32; 128 -> 128 at 64^2, 272 CTAs 42 us, 304 40.
int wgrad_splits(int n, int h, int w, int cin, int cout) {
  const int cc = cin % 64 == 0 ? 64 : cin % 32 == 0 ? 32 : 16, nt = cout % 64 == 0 ? 64 : cout % 32 == 0 ? 32 : 16;
  const int tx = wgrad_tile(w), ty = kWgPix / tx, ktiles = (9 * cin + 127) / 128;
  const long long np = (long long)n * h * w, tiles = (long long)n * ((h + ty - 1) / ty) * ((w + tx - 1) / tx);
  const int ctas = (cin / cc) * (cout / nt), wave = 3 * nt * (cc == 64 ? 2 : 1) > 256 ? 152 : 304;
  const long long least = std::max(1ll, std::min(np / 256, (608ll + ktiles - 1) / ktiles));
  const long long splits = (least * ctas + wave - 1) / wave * wave / ctas;
  return (int)std::min(std::max(splits, least), tiles);
}

}  // namespace mcx

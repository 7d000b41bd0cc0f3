// Volumes with clearance (VOX_HOP, VOX_HOP2): which voxels ahead of a voxel hold the same
// material and density, per direction octant, so that a march takes all the
// midpoints inside a uniform cube from one word (mc_device.cuh, Hop).
//
// A word holds an 8-bit palette index (the volume's distinct (material,
// density) pairs, at most 256) and a 3-bit code c per octant o: the cube that
// starts at the voxel and extends r = 2^c - 1 voxels along each axis in the
// octant's direction is uniform.  Octant bit a is set where the ray runs toward
// smaller coordinates of axis a.  A volume with more pairs keeps the codes in a
// second word beside the voxel's own (VOX_HOP2).
//
// Everything is built from bit masks along x.  A cell is the 2 x 2 x 2 cube of
// voxels at v .. v + 1; level r of a voxel says that the r^3 cells from v on
// are uniform, which makes the voxels v .. v + r uniform, and level 2r + 1 is
// the conjunction of level r at the offsets {0, r, r + 1} per axis.  An octant
// running toward smaller coordinates reads the level r bits farther down, so
// the seven levels serve all eight octants: about 2 words of traffic per 32
// voxels and level instead of a distance per voxel and octant.
#include <stdint.h>

#include <algorithm>

#include "mc_device.cuh"

namespace mcx {
namespace {

constexpr int kLevels = 7;              // r = 1, 3, 7, 15, 31, 63, 127
constexpr int kKeys = kMaxMat << 15;    // material x FP16 density without its sign

// Material and density as one number; -0 is 0.
__device__ __forceinline__ uint32_t voxel_key(uint32_t mat, uint32_t rho) { return (mat << 15) | (rho & 0x7FFFu); }

// One pass over a volume's arrays: whether every material id is below n_mat and
// every density a finite, non-negative binary16 (out->bad), the x-neighbour
// pairs of different materials (out->changes), and a mark for every key that
// occurs.  VEC voxels per thread and step (8: one 8-byte and one 16-byte load,
// for arrays aligned to them).  Marks are kept per block in shared memory and
// merged at its end; a block that has seen more keys than a palette holds says
// so (out->pairs) and stops marking, so that a volume with a density of its own
// in every voxel is read at the speed of its loads (a noisy 256^3 and 128^3:
// 160 -> 46 us together).
constexpr int kScanWords = kKeys / 32;
template <int VEC>
__global__ void __launch_bounds__(256) k_scan_volume(const uint8_t* __restrict__ mat, const uint16_t* __restrict__ rho,
                                                     size_t n, uint32_t nx, int n_mat, VolumeScan* out,
                                                     uint32_t* __restrict__ seen) {
  __shared__ uint32_t marks[kScanWords];
  __shared__ volatile uint32_t n_keys;
  for (int i = threadIdx.x; i < kScanWords; i += blockDim.x) marks[i] = 0u;
  if (threadIdx.x == 0) n_keys = 0u;
  __syncthreads();
  uint32_t last = 0xFFFFFFFFu, changes = 0;
  int bad = 0;
  auto voxel = [&](uint32_t m, uint32_t h) {
    const bool wrong = m >= (uint32_t)n_mat || h > 0x8000u || (h & 0x7C00u) == 0x7C00u;
    bad |= wrong;
    const uint32_t key = voxel_key(m, h);
    if (wrong || key == last || n_keys > (uint32_t)kMaxPalette) return;
    last = key;
    const uint32_t bit = 1u << (key & 31);
    if (!(marks[key >> 5] & bit) && !(atomicOr(&marks[key >> 5], bit) & bit)) atomicAdd((uint32_t*)&n_keys, 1u);
  };
  const size_t stride = (size_t)gridDim.x * blockDim.x * VEC;
  for (size_t i = ((size_t)blockIdx.x * blockDim.x + threadIdx.x) * VEC; i < n; i += stride) {
    uint32_t x = (uint32_t)(i % nx);
    uint32_t m[VEC], h[VEC];
    const int k_end = (int)min((size_t)VEC, n - i);
    if (VEC == 8 && k_end == VEC) {
      const uint2 a = __ldg(reinterpret_cast<const uint2*>(mat + i));
      const uint4 b = __ldg(reinterpret_cast<const uint4*>(rho + i));
      const uint32_t aw[2] = {a.x, a.y}, bw[4] = {b.x, b.y, b.z, b.w};
#pragma unroll
      for (int k = 0; k < VEC; ++k) {
        m[k] = (aw[k >> 2] >> (8 * (k & 3))) & 255u;
        h[k] = (bw[(k >> 1) & 3] >> (16 * (k & 1))) & 0xFFFFu;
      }
    } else {
#pragma unroll
      for (int k = 0; k < VEC; ++k) {
        m[k] = k < k_end ? mat[i + k] : 0u;
        h[k] = k < k_end ? rho[i + k] : 0u;
      }
    }
    const uint32_t after = i + VEC < n ? mat[i + VEC] : 0u;  // the voxel after this group's last
#pragma unroll
    for (int k = 0; k < VEC; ++k) {
      if (k < k_end) {
        voxel(m[k], h[k]);
        const uint32_t next = k + 1 < k_end ? m[(k + 1) % VEC] : after;
        changes += (x + 1 != nx && next != m[k]) ? 1u : 0u;
        if (++x == nx) x = 0;
      }
    }
  }
  for (int o = 16; o > 0; o >>= 1) changes += __shfl_down_sync(0xffffffffu, changes, o);
  if ((threadIdx.x & 31) == 0 && changes) atomicAdd(&out->changes, (unsigned long long)changes);
  if (__syncthreads_or(bad) && threadIdx.x == 0) atomicOr(&out->bad, 1u);
  if (n_keys > (uint32_t)kMaxPalette) {  // uniform: nothing is marked after the barrier
    if (threadIdx.x == 0) atomicMax(&out->pairs, n_keys);
    return;
  }
  for (int i = threadIdx.x; i < kScanWords; i += blockDim.x) {
    const uint32_t w = marks[i];
    if (w & ~__ldcg(seen + i)) atomicOr(seen + i, w);
  }
}

// Numbers the marked keys in order (one block): pal[index] the voxel word,
// map[key] the index, *count the number of keys (more than kMaxPalette: no palette).
__global__ void __launch_bounds__(1024) k_palette(const uint32_t* __restrict__ seen, uint32_t* __restrict__ pal,
                                                  uint8_t* __restrict__ map, uint32_t* __restrict__ count) {
  __shared__ uint32_t part[1024];
  constexpr int kWords = kKeys / 32 / 1024;
  if (*count > (uint32_t)kMaxPalette) return;  // found by the scan
  uint32_t n = 0;
  for (int k = 0; k < kWords; ++k) n += __popc(seen[threadIdx.x * kWords + k]);
  part[threadIdx.x] = n;
  __syncthreads();
  for (int o = 1; o < 1024; o <<= 1) {
    const uint32_t v = threadIdx.x >= o ? part[threadIdx.x - o] : 0u;
    __syncthreads();
    part[threadIdx.x] += v;
    __syncthreads();
  }
  // every thread is past the test above (the barriers)
  if (threadIdx.x == 1023) *count = part[1023];
  uint32_t at = part[threadIdx.x] - n;
  for (int k = 0; k < kWords; ++k)
    for (uint32_t m = seen[threadIdx.x * kWords + k]; m; m &= m - 1) {
      if (at >= kMaxPalette) return;
      const uint32_t key = (threadIdx.x * kWords + k) * 32 + (__ffs(m) - 1);
      pal[at] = (key & 0x7FFFu) | ((key >> 15) << 16);
      map[key] = (uint8_t)at++;
    }
}

// Palette indices, or voxel words beside an empty word, over the padded grid (border voxels repeat the nearest edge
// voxel).
template <int LAYOUT>
__global__ void __launch_bounds__(256) k_pack_clearance(const uint8_t* __restrict__ mat, const uint16_t* __restrict__ rho,
                                                      VolumeView v, const uint8_t* __restrict__ map,
                                                      uint32_t* __restrict__ out) {
  // 32-bit indices: the packed volume has fewer than 2^31 words
  const uint32_t n = (uint32_t)v.words;
  for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    const uint32_t r = i / (uint32_t)v.px;
    const int px = (int)(i - r * (uint32_t)v.px), pz = (int)(r / (uint32_t)v.py), py = (int)(r - pz * (uint32_t)v.py);
    const int ix = min(max(px - 1, 0), v.nx - 1), iy = min(max(py - 1, 0), v.ny - 1), iz = min(max(pz - 1, 0), v.nz - 1);
    const size_t src = ((size_t)iz * v.ny + iy) * v.nx + ix;
    if (LAYOUT == VOX_HOP2)
      reinterpret_cast<uint2*>(out)[i] = make_uint2((uint32_t)(rho[src] & 0x7FFFu) | ((uint32_t)mat[src] << 16), 0u);
    else
      out[i] = map[voxel_key(mat[src], rho[src])];
  }
}

// Level 1 over the padded grid, from the volume's own arrays, so that a volume is looked over before any words are made
// for it: cell (x, y, z) is uniform; cells past the last voxel compare the
// voxels there are, bits past the row are set.  Counts the mixed cells.  A warp
// walks kZRun planes of one row word: a plane's 2 x 2 patch is reduced to its
// value (or "mixed") once and serves the cells below and above it, with the
// x + 1 neighbours from a shuffle: 2 voxels read per voxel.
constexpr int kZRun = 8;
__global__ void __launch_bounds__(256) k_cells(const uint8_t* __restrict__ mat, const uint16_t* __restrict__ rho, int nx,
                                               int ny, int nz, int wpr, uint32_t* __restrict__ bits,
                                               unsigned long long* mixed) {
  const int px = nx + 2, py = ny + 2, pz = nz + 2;
  const uint32_t runs = (uint32_t)((pz + kZRun - 1) / kZRun);
  const uint32_t work = (uint32_t)wpr * (uint32_t)py * runs;
  const int lane = threadIdx.x & 31;
  uint32_t n = 0;
  for (uint32_t i = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; i < work; i += (gridDim.x * blockDim.x) >> 5) {
    const uint32_t t = i / (uint32_t)wpr, wi = i - t * (uint32_t)wpr;
    const int y = (int)(t % (uint32_t)py), z0 = (int)(t / (uint32_t)py) * kZRun, z1 = min(z0 + kZRun, pz);
    // border voxels repeat the nearest edge voxel
    const int x = (int)wi * 32 + lane, xc = min(max(x - 1, 0), nx - 1), xe = min(x, nx - 1);
    const int y0 = min(max(y - 1, 0), ny - 1), y1 = min(y, ny - 1);
    constexpr uint32_t kMixed = 0xFFFFFFFFu;  // no voxel's key
    auto key = [&](size_t at) { return voxel_key(__ldg(mat + at), __ldg(rho + at)); };
    auto patch = [&](int z) -> uint32_t {
      const size_t zs = (size_t)min(max(z - 1, 0), nz - 1) * ny, r0 = (zs + y0) * nx, r1 = (zs + y1) * nx;
      const uint32_t a = key(r0 + xc), b = key(r1 + xc);
      uint32_t an = __shfl_down_sync(0xffffffffu, a, 1), bn = __shfl_down_sync(0xffffffffu, b, 1);
      if (lane == 31) {
        an = key(r0 + xe);
        bn = key(r1 + xe);
      }
      return a == b && a == an && a == bn ? a : kMixed;
    };
    uint32_t here = patch(z0);
    for (int z = z0; z < z1; ++z) {
      const uint32_t above = patch(min(z + 1, pz - 1));
      const uint32_t m = __ballot_sync(0xffffffffu, x >= px || (here != kMixed && here == above));
      if (lane == 0) {
        bits[((size_t)z * py + y) * wpr + wi] = m;
        n += 32 - __popc(m);
      }
      here = above;
    }
  }
  if (lane == 0 && n) atomicAdd(mixed, (unsigned long long)n);
}

// 32 bits of a row from bit x on (x >= 0; past the row all set).
__device__ __forceinline__ uint32_t row_bits(const uint32_t* __restrict__ row, int wpr, int x) {
  const int wi = x >> 5;
  const uint32_t lo = wi < wpr ? __ldg(row + wi) : 0xFFFFFFFFu;
  const uint32_t hi = wi + 1 < wpr ? __ldg(row + wi + 1) : 0xFFFFFFFFu;
  return __funnelshift_r(lo, hi, x & 31);
}

// Level 2r + 1 from level r (rows and planes past the volume restrict nothing).
__global__ void __launch_bounds__(256) k_level(const uint32_t* __restrict__ in, int r, int py, int pz, int wpr,
                                               uint32_t* __restrict__ out) {
  const uint32_t words = (uint32_t)wpr * (uint32_t)py * (uint32_t)pz;
  for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < words; i += gridDim.x * blockDim.x) {
    const uint32_t row = i / (uint32_t)wpr;
    const int x = (int)(i - row * (uint32_t)wpr) * 32, z = (int)(row / (uint32_t)py), y = (int)(row - z * (uint32_t)py);
    uint32_t m = 0xFFFFFFFFu;
#pragma unroll
    for (int a = 0; a < 3; ++a)
#pragma unroll
      for (int b = 0; b < 3; ++b) {
        const int zz = z + (a == 0 ? 0 : r + a - 1), yy = y + (b == 0 ? 0 : r + b - 1);
        if (m && zz < pz && yy < py) {
          const uint32_t* q = in + ((size_t)zz * py + yy) * wpr;
          m &= row_bits(q, wpr, x) & row_bits(q, wpr, x + r) & row_bits(q, wpr, x + r + 1);
        }
      }
    out[i] = m;
  }
}

// The octant codes of every voxel: how many levels hold from the voxel on (or,
// along an axis the octant runs down, from r voxels lower; cubes that would
// start below the volume start at its first voxel, which asks for more).  A
// lane counts the levels of the 32 voxels of one row word for all octants at
// once, three bit planes per octant, stopping at the first level that no voxel
// of its warp reaches; the planes are turned into words in shared memory, from
// where the warp writes row by row.
constexpr int kCodeWarps = 4;
template <int LAYOUT>
__global__ void __launch_bounds__(32 * kCodeWarps) k_codes(const uint32_t* __restrict__ bits, size_t level_words, int px,
                                                           int py, int pz, int wpr, uint32_t* __restrict__ vox) {
  // [row word of the warp][bit plane, 24 used]: 16-byte rows read by all lanes at once
  __shared__ __align__(16) uint32_t planes[kCodeWarps][32][28];
  const uint32_t words = (uint32_t)wpr * (uint32_t)py * (uint32_t)pz;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const uint32_t step = gridDim.x * 32 * kCodeWarps;
  for (uint32_t base = (blockIdx.x * kCodeWarps + warp) * 32; base < words; base += step) {
    const uint32_t i = min(base + lane, words - 1);
    const uint32_t row = i / (uint32_t)wpr;
    const int x = (int)(i - row * (uint32_t)wpr) * 32, z = (int)(row / (uint32_t)py), y = (int)(row - z * (uint32_t)py);
    uint32_t b0[8] = {}, b1[8] = {}, b2[8] = {};
    for (int l = 0; l < kLevels; ++l) {
      const int r = (2 << l) - 1;
      const uint32_t* lv = bits + (size_t)l * level_words;
      const int ym = max(y - r, 0), zm = max(z - r, 0);
      uint32_t any = 0;
#pragma unroll
      for (int o = 0; o < 8; o += 2) {
        const uint32_t* q = lv + ((size_t)((o & 4) ? zm : z) * py + ((o & 2) ? ym : y)) * wpr;
        const uint32_t up = __ldg(q + (x >> 5));
        // bits x - r .. x - r + 31 of the row, bit 0 of the row where that is negative
        uint32_t down;
        if (x >= r) {
          down = row_bits(q, wpr, x - r);
        } else {
          const uint32_t w0 = __ldg(q), first = (w0 & 1u) ? 0xFFFFFFFFu : 0u;
          const int gap = r - x;  // that many bits lie before the row
          down = gap >= 32 ? first : ((w0 << gap) | (first >> (32 - gap)));
        }
#pragma unroll
        for (int d = 0; d < 2; ++d) {
          const uint32_t p = d ? down : up;
          const uint32_t c0 = b0[o + d] & p, c1 = b1[o + d] & c0;
          b0[o + d] ^= p;
          b1[o + d] ^= c0;
          b2[o + d] ^= c1;
          any |= p;
        }
      }
      if (!__any_sync(0xffffffffu, any)) break;
    }
    __syncwarp();
#pragma unroll
    for (int o = 0; o < 8; ++o) {
      planes[warp][lane][3 * o] = b0[o];
      planes[warp][lane][3 * o + 1] = b1[o];
      planes[warp][lane][3 * o + 2] = b2[o];
    }
    __syncwarp();
    const int count = (int)min(32u, words - base);
    for (int k = 0; k < count; ++k) {  // row word k of the warp: lane = voxel
      const uint32_t j = base + k, jr = j / (uint32_t)wpr;
      const int jx = (int)(j - jr * (uint32_t)wpr) * 32 + lane;
      uint32_t codes = 0;
#pragma unroll
      for (int b = 0; b < 24; b += 4) {
        const uint4 q = *reinterpret_cast<const uint4*>(&planes[warp][k][b]);
        codes |= (((q.x >> lane) & 1u) | (((q.y >> lane) & 1u) << 1) | (((q.z >> lane) & 1u) << 2) |
                  (((q.w >> lane) & 1u) << 3)) << b;
      }
      if (jx < px) {
        const size_t at = (size_t)jr * px + jx;
        if (LAYOUT == VOX_HOP2) vox[2 * at + 1] = codes << 8;
        else vox[at] |= codes << 8;
      }
    }
  }
}

size_t level_words(int px, int py, int pz) { return (size_t)((px + 31) / 32) * py * pz; }

int grid_of(size_t threads) {
  const size_t b = (threads + 255) / 256;
  return (int)(b < 152 * 32 ? (b > 0 ? b : 1) : 152 * 32);
}

// Scratch: the scan's results, the key marks, the map of the marked keys, the levels.
constexpr size_t kScanBytes = 64;
static_assert(sizeof(VolumeScan) <= kScanBytes, "scan results");
uint32_t* scratch_seen(void* scratch) { return reinterpret_cast<uint32_t*>(static_cast<unsigned char*>(scratch) + kScanBytes); }
uint8_t* scratch_map(void* scratch) { return static_cast<unsigned char*>(scratch) + kScanBytes + kKeys / 8; }
uint32_t* scratch_levels(void* scratch) { return reinterpret_cast<uint32_t*>(scratch_map(scratch) + kKeys); }

cudaError_t read_scan(void* scratch, VolumeScan* out, cudaStream_t s) {
  cudaError_t e = cudaMemcpyAsync(out, scratch, sizeof(VolumeScan), cudaMemcpyDeviceToHost, s);
  if (e == cudaSuccess) e = cudaStreamSynchronize(s);
  return e;
}

}  // namespace

size_t scan_scratch_bytes() { return kScanBytes + kKeys / 8 + kKeys; }
size_t cells_scratch_bytes(int nx, int ny, int nz) {
  return scan_scratch_bytes() + level_words(nx + 2, ny + 2, nz + 2) * 4;
}
size_t clearance_scratch_bytes(int nx, int ny, int nz) {
  return scan_scratch_bytes() + (size_t)kLevels * level_words(nx + 2, ny + 2, nz + 2) * 4;
}

cudaError_t scan_volume(const uint8_t* mat, const uint16_t* rho, int nx, int ny, int nz, int n_mat, void* scratch,
                        uint32_t* pal, VolumeScan* out, cudaStream_t s) {
  const size_t n = (size_t)nx * ny * nz;
  cudaError_t e = cudaMemsetAsync(scratch, 0, kScanBytes + kKeys / 8, s);
  if (e != cudaSuccess) return e;
  auto* scan = static_cast<VolumeScan*>(scratch);
  if (((uintptr_t)mat & 7) == 0 && ((uintptr_t)rho & 15) == 0)
    k_scan_volume<8><<<std::min(grid_of((n + 7) / 8), 152 * 6), 256, 0, s>>>(mat, rho, n, (uint32_t)nx, n_mat, scan,
                                                                             scratch_seen(scratch));
  else
    k_scan_volume<1><<<std::min(grid_of(n), 152 * 6), 256, 0, s>>>(mat, rho, n, (uint32_t)nx, n_mat, scan,
                                                                   scratch_seen(scratch));
  k_palette<<<1, 1024, 0, s>>>(scratch_seen(scratch), pal, scratch_map(scratch), &scan->pairs);
  e = cudaGetLastError();
  return e == cudaSuccess ? read_scan(scratch, out, s) : e;
}

cudaError_t mixed_cells(const uint8_t* mat, const uint16_t* rho, int nx, int ny, int nz, void* scratch, double* share,
                        cudaStream_t s) {
  const int wpr = (nx + 2 + 31) / 32;
  auto* scan = static_cast<VolumeScan*>(scratch);
  cudaError_t e = cudaMemsetAsync(&scan->mixed, 0, sizeof(scan->mixed), s);
  if (e != cudaSuccess) return e;
  k_cells<<<grid_of(level_words(nx + 2, ny + 2, (nz + 2 + kZRun - 1) / kZRun) * 32), 256, 0, s>>>(
      mat, rho, nx, ny, nz, wpr, scratch_levels(scratch), &scan->mixed);
  e = cudaGetLastError();
  VolumeScan h = {};
  if (e == cudaSuccess) e = read_scan(scratch, &h, s);
  *share = (double)h.mixed / ((double)(nx + 2) * (ny + 2) * (nz + 2));
  return e;
}

cudaError_t build_clearance(const uint8_t* mat, const uint16_t* rho, int nx, int ny, int nz, int layout, void* scratch,
                            uint32_t* vox, cudaStream_t s) {
  VolumeView v;
  padded_dims(nx, ny, nz, layout, &v);
  uint32_t* bits = scratch_levels(scratch);
  const size_t lw = level_words(v.px, v.py, v.pz);
  const int wpr = (v.px + 31) / 32, gp = grid_of((size_t)v.words);
  if (layout == VOX_HOP2) k_pack_clearance<VOX_HOP2><<<gp, 256, 0, s>>>(mat, rho, v, scratch_map(scratch), vox);
  else k_pack_clearance<VOX_HOP><<<gp, 256, 0, s>>>(mat, rho, v, scratch_map(scratch), vox);
  for (int l = 0; l + 1 < kLevels; ++l)
    k_level<<<grid_of(lw), 256, 0, s>>>(bits + l * lw, (2 << l) - 1, v.py, v.pz, wpr, bits + (l + 1) * lw);
  const size_t blocks = (lw + 32 * kCodeWarps - 1) / (32 * kCodeWarps);
  const int g = (int)(blocks < 152 * 32 ? blocks : 152 * 32);
  if (layout == VOX_HOP2) k_codes<VOX_HOP2><<<g, 32 * kCodeWarps, 0, s>>>(bits, lw, v.px, v.py, v.pz, wpr, vox);
  else k_codes<VOX_HOP><<<g, 32 * kCodeWarps, 0, s>>>(bits, lw, v.px, v.py, v.pz, wpr, vox);
  return cudaGetLastError();
}

}  // namespace mcx

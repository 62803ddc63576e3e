// Front-to-back alpha compositing of the primitives (the consumer of the
// per-primitive colours) and its backward to the colours and opacities:
// nasg_raster_forward / nasg_raster_backward.
//
// Sec. 3.1: C(r) = sum_i T_i alpha_i c_i, alpha_i = sigma_i rho_i,
// T_i = prod_{j<i} (1 - alpha_j), with rho_i the primitive's Gaussian kernel
// projected onto the image plane. Rules (the compositing conventions of the
// Gaussian-splatting rasterizer the paper builds on):
//   camera      p = R (mu - centre), rows (right, up, forward); x = cx + fx p_x/p_z,
//               y = cy - fy p_y/p_z; pixel (i, j) sampled at (i + 0.5, j + 0.5);
//               p_z <= near is not drawn;
//   projection  Sigma' = J R Sigma R^T J^T + 0.3 I (local affine approximation,
//               screen-space low-pass), Sigma = Rq diag(s^2) Rq^T;
//   alpha       min(0.99, sigma exp(-q/2)), q = delta^T Sigma'^-1 delta; a primitive
//               contributes to a pixel iff alpha >= 1/255;
//   order       by p_z, ties by primitive index;
//   stop        a pixel stops before the contribution that would take T below 1e-4.
//
// Pipeline (all on one stream): per-primitive projection, footprint (a square holding every
// pixel centre where alpha >= 1/255 can hold, so the image does not depend on the binning),
// and within it, row by row, the tiles that the ellipse can reach, with the digit counts
// of both sorts; a stable LSD radix sort of the drawn primitives by depth (four passes,
// one launch each); an exclusive scan, in that order, of the tiles each primitive reaches; a
// stable radix sort of the (tile, index) pairs by tile, whose first pass lists its pairs itself
// and whose last pass notes the tiles' ranges (so each tile's list is in depth order,
// ties by index); then one block per 16 x 16 tile, whose warps own
// sub-tiles (8 x 8 pixels, two per lane, or 8 x 4 pixels, one per lane): batches of
// primitives are staged in shared memory, the staging threads note which sub-tiles each
// primitive's alpha >= 1/255 ellipse can reach, and each warp walks the ones that reach
// its own. The backward walks each pixel's list back to front (T recovered by division),
// reduces the four per-primitive gradients over the warp in six shuffles, over the tile's
// warps in shared memory, and adds them with one atomic per tile, value and primitive. The
// forward reads the footprint squares' pair total once on the host (the capacity check and the
// size of the pair sort), waiting only for the projection.
#include <algorithm>
#include <atomic>
#include <cmath>
#include <cstdint>
#include <thread>

#include "nasg_cover.h"
#include "nasg_host.h"
#include "nasg_list.h"
#include "nasg_sort.cuh"
#include "nasg_vec.cuh"

namespace nasg {
namespace raster {

constexpr int kTile = 16;
constexpr int kTilePixels = kTile * kTile;
constexpr int kBlock = 256;
constexpr int kDepthPasses = 4;                   // 8-bit digits of the depth key
constexpr int kMaxTilePasses = 4;                 // tile keys: two digits for columns, two for rows
constexpr int kScanItems = 8;                     // primitives per thread of the offset scan
constexpr int kStartGrain = 1024;                 // pairs per entry of the table of first primitives
constexpr float kAlphaMin = 1.f / 255.f;
constexpr float kAlphaMax = 0.99f;
constexpr float kTMin = 1e-4f;
constexpr float kLowPass = 0.3f;
constexpr float kLog2e = 1.44269504088896341f;
constexpr float kExpScale = -0.5f * kLog2e;       // rho = 2^(q kExpScale)

// What the rendering kernels read of a projected primitive, one 32-byte sector:
// {mean x, mean y, A, 2B}, {C, sigma, cull, 0} with q = A dx^2 + 2B dx dy + C dy^2.
// cull: a primitive may be left out of a pixel set whose smallest q is above it (no
// pixel there can reach alpha >= 1/255); infinity where that is not certain in FP32.
struct Splat {
  float4 a, b;
};

struct Cam {
  float r[9], c[3], fx, fy, cx, cy, near_z;
  int w, h, tx, ty;
};

// First words of the workspace, zeroed by each forward.
struct Header {
  unsigned long long pairs64;             // pairs of the footprint squares (what n_pairs reports)
  uint32_t pairs;                         // pairs listed: tiles the ellipses can reach
  uint32_t drawn;                         // primitives that reach a tile
  uint32_t failed;                        // a bounded wait gave up: no list may be trusted
  uint32_t projected;                     // blocks of the projection that are done
  uint32_t tickets[kDepthPasses + 1 + kMaxTilePasses];
  uint32_t depth_hist[kDepthPasses][sort::kBins];
  uint32_t tile_hist[kMaxTilePasses][sort::kBins];
};

// Shape of a sort block. A pass's blocks learn their places one after the other, so many small
// blocks cost more than their entries; few large ones leave SMs idle. 256 threads x 4 entries
// up to the lines below, 512 x 16 (two blocks per SM) above. Forward at 320 x 180, small /
// large depth blocks: 3e5 primitives 205 / 215 us, 5e5 291 / 260, 8e5 347 / 288; pairs (of the
// squares) 8.8e5 173 / 183 us, 1.1e6 191 / 189, 1.5e6 221 / 222; 1.39e7 pairs (1080p) list and
// sort 476 us small, 226 us at 256 x 16, 201 us at 512 x 16, 228 us at 1024 x 16.
constexpr int kLargeThreads = 512, kLargeItems = 16, kSmallThreads = 256, kSmallItems = 4;
constexpr int64_t kLargeDepth = 400000, kLargePairs = 1000000;
__host__ __device__ inline int64_t sort_blocks(int64_t m, int64_t line) {
  const int64_t per = m > line ? kLargeThreads * kLargeItems : kSmallThreads * kSmallItems;
  return (m + per - 1) / per;
}
// the most blocks that any m <= cap takes
inline int64_t sort_blocks_max(int64_t cap, int64_t line) {
  return std::max(sort_blocks(cap, line), sort_blocks(cap < line ? cap : line, line));
}

// Workspace layout (byte offsets, each 256-aligned), from n, tiles, pixels and the pair capacity.
// [header, head_end) is zeroed by every forward; pair_states as far as the pairs need it.
struct Layout {
  size_t header, ranges, scan_states, depth_states, head_end, pair_states, splat, rows, rect, reach, offsets, starts,
      dkeys0, dkeys1, order0, order1, keys0, keys1, vals0, vals1, ncontrib, total;
};

inline size_t align256(size_t x) { return (x + 255) & ~size_t(255); }

inline Layout layout(int64_t n, int64_t tiles, int64_t pixels, int64_t cap) {
  Layout L{};
  size_t o = 0;
  auto take = [&](size_t bytes) { const size_t at = o; o = align256(o + bytes); return at; };
  const size_t state = sizeof(unsigned long long);
  L.header = take(sizeof(Header));
  L.ranges = take(size_t(tiles) * sizeof(uint2));
  L.scan_states = take(size_t(n / (kBlock * kScanItems) + 1) * state);
  L.depth_states = take(size_t(sort_blocks(n, kLargeDepth)) * sort::kBins * state);
  L.head_end = o;
  L.pair_states = take(size_t(sort_blocks_max(cap, kLargePairs)) * sort::kBins * state);
  L.splat = take(size_t(n) * sizeof(Splat));
  L.rows = take(size_t(n) * sizeof(CoverRows));
  L.rect = take(size_t(n) * sizeof(uint2));
  L.reach = take(size_t(n) * sizeof(uint32_t));
  L.offsets = take(size_t(n) * sizeof(uint32_t));
  L.starts = take(size_t(cap / kStartGrain + 1) * sizeof(uint32_t));
  L.dkeys0 = take(size_t(n) * sizeof(uint32_t));
  L.dkeys1 = take(size_t(n) * sizeof(uint32_t));
  L.order0 = take(size_t(n) * sizeof(uint32_t));
  L.order1 = take(size_t(n) * sizeof(uint32_t));
  L.keys0 = take(size_t(cap) * sizeof(uint32_t));
  L.keys1 = take(size_t(cap) * sizeof(uint32_t));
  L.vals0 = take(size_t(cap) * sizeof(uint32_t));
  L.vals1 = take(size_t(cap) * sizeof(uint32_t));
  L.ncontrib = take(size_t(pixels) * sizeof(uint32_t));
  L.total = o;
  return L;
}

// A tile's sort key is its row above its column, ty << x_bits | tx, in digits of at most 8 bits
// that do not straddle the two unless the whole key fits one digit: then the tiles of one row of a
// footprint are one run of the lowest digit and share the rest (but for images over 4096 pixels).
struct TileDigits {
  int x_bits, passes;
  int shift[kMaxTilePasses], bits[kMaxTilePasses];
};
inline TileDigits tile_digits(int tiles_x, int tiles_y) {
  auto bits_for = [](int n) {
    int b = 0;
    while ((1 << b) < n) ++b;
    return b;
  };
  TileDigits d{};
  d.x_bits = bits_for(tiles_x);
  const int y_bits = bits_for(tiles_y);
  auto add = [&](int from, int width) {
    const int parts = (width + 7) / 8;
    for (int at = 0, p = 0; p < parts; ++p) {
      const int w = (width - at + parts - p - 1) / (parts - p);
      d.shift[d.passes] = from + at;
      d.bits[d.passes++] = w;
      at += w;
    }
  };
  if (d.x_bits + y_bits <= 8) {
    add(0, std::max(1, d.x_bits + y_bits));
  } else {
    add(0, d.x_bits);
    add(d.x_bits, y_bits);
  }
  return d;
}

// ---------------------------------------------------------------------------
// Projection and footprint
// ---------------------------------------------------------------------------

// Digit counts of a block's primitives, kept in shared memory until the block is done.
struct Counts {
  uint32_t depth[kDepthPasses][sort::kBins];
  uint32_t tile[kMaxTilePasses][sort::kBins + 1];  // [0] as differences of neighbouring digits
};

// Adds 1 to `bin` for every lane of the warp (bin 256 for none), one addition per distinct bin.
__device__ __forceinline__ void count_merged(uint32_t* hist, uint32_t bin, int lane) {
  const uint32_t peers = __match_any_sync(0xffffffffu, bin);
  if (bin < uint32_t(sort::kBins) && lane == __ffs(int(peers)) - 1) atomicAdd(hist + bin, uint32_t(__popc(peers)));
}

// Adds the digits of the consecutive tile keys [t0, t1], all of one tile row: the lowest digit as
// the ends of its runs (a prefix sum at the end of the kernel turns them into counts), the others
// run by run.
__device__ __forceinline__ void count_tiles(Counts& c, uint32_t t0, uint32_t t1, const TileDigits& td) {
  const uint32_t bins = 1u << td.bits[0], mask = bins - 1u;
  const uint32_t len = t1 - t0 + 1u, s0 = t0 & mask, rest = len & mask;
  if (len > mask) atomicAdd(&c.tile[0][0], len >> td.bits[0]);  // whole turns: every digit
  if (rest) {
    atomicAdd(&c.tile[0][s0], 1u);
    const bool wraps = s0 + rest > bins;
    atomicSub(&c.tile[0][s0 + rest - (wraps ? bins : 0u)], 1u);
    if (wraps) atomicAdd(&c.tile[0][0], 1u);
  }
  for (int j = 1; j < td.passes; ++j) {
    const int shift = td.shift[j];
    const uint32_t digits = (1u << td.bits[j]) - 1u;
    for (uint32_t h = t0 >> shift; h <= t1 >> shift; ++h) {
      const uint32_t lo = max(t0, h << shift), hi = min(t1, ((h + 1u) << shift) - 1u);
      atomicAdd(&c.tile[j][h & digits], hi - lo + 1u);
    }
  }
}

// Where the projection leaves its pair total for the host: two page-locked words, the total and
// then the call's number (a late write of an earlier call does not match).
struct HostTotal {
  unsigned long long pairs;
  unsigned long long call;
};

// Programmatic dependent launch: a kernel of the forward's chain lets the next one start when its
// blocks have only their results to write, and reads or writes nothing before its predecessor
// has finished, so that a launch's latency passes meanwhile: the ten launches of a 640 x 360 preview of
// 2e4 primitives take 124 us one by one and 112 us chained. Allowed at the start of the blocks
// instead, the next pass's blocks crowd onto the SMs that the running pass leaves free (two of
// 512 threads on one, none on another): 8e5 primitives at 320 x 180 337 us instead of 288 us.
__device__ __forceinline__ void chain_next() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void chain_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

struct ProjectArgs {
  int64_t n;
  const float *means, *scales, *quats, *opacity;
  Cam cam;
  TileDigits td;
  Splat* splat;
  CoverRows* rows;
  uint2* rect;      // tile columns x0 | x1 << 16, rows y0 | y1 << 16
  uint32_t* reach;  // tiles reached
  uint32_t* dkey;  // depth bits, kNone where nothing is drawn
  Header* hdr;
  HostTotal* host;
  unsigned long long call;
};

// Footprint of primitive i: the number of tiles of its square (*square), the tiles its ellipse
// reaches (returned, and counted by digit).
__device__ __forceinline__ uint32_t project_one(const ProjectArgs& a, int64_t i, Counts& counts, uint32_t* square,
                                                uint32_t* key) {
  const Cam& cam = a.cam;
  const float* __restrict__ means = a.means;
  const float* __restrict__ scales = a.scales;
  const float* __restrict__ quats = a.quats;
  uint32_t count = 0;
  *square = 0;
  const float mx = means[3 * i] - cam.c[0], my = means[3 * i + 1] - cam.c[1], mz = means[3 * i + 2] - cam.c[2];
  const float px = cam.r[0] * mx + cam.r[1] * my + cam.r[2] * mz;
  const float py = cam.r[3] * mx + cam.r[4] * my + cam.r[5] * mz;
  const float pz = cam.r[6] * mx + cam.r[7] * my + cam.r[8] * mz;
  const float sig = a.opacity[i];
  if (pz > cam.near_z && sig * 255.f > 1.f) {
    const float iz = 1.f / pz;
    const float u = cam.cx + cam.fx * px * iz;
    const float v = cam.cy - cam.fy * py * iz;
    // J (2x3): rows (fx/z, 0, -fx x/z^2), (0, -fy/z, fy y/z^2); M = J R
    const float j00 = cam.fx * iz, j02 = -cam.fx * px * iz * iz;
    const float j11 = -cam.fy * iz, j12 = cam.fy * py * iz * iz;
    float m0[3], m1[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      m0[c] = j00 * cam.r[c] + j02 * cam.r[6 + c];
      m1[c] = j11 * cam.r[3 + c] + j12 * cam.r[6 + c];
    }
    // Sigma = Rq diag(s^2) Rq^T from the normalised quaternion (w, x, y, z)
    float qw = quats[4 * i], qx = quats[4 * i + 1], qy = quats[4 * i + 2], qz = quats[4 * i + 3];
    const float qn = rsqrtf(qw * qw + qx * qx + qy * qy + qz * qz);
    qw *= qn; qx *= qn; qy *= qn; qz *= qn;
    const float R[9] = {1.f - 2.f * (qy * qy + qz * qz), 2.f * (qx * qy - qw * qz), 2.f * (qx * qz + qw * qy),
                        2.f * (qx * qy + qw * qz), 1.f - 2.f * (qx * qx + qz * qz), 2.f * (qy * qz - qw * qx),
                        2.f * (qx * qz - qw * qy), 2.f * (qy * qz + qw * qx), 1.f - 2.f * (qx * qx + qy * qy)};
    const float s0 = scales[3 * i], s1 = scales[3 * i + 1], s2 = scales[3 * i + 2];
    const float ss[3] = {s0 * s0, s1 * s1, s2 * s2};
    // A = M Rq (2x3); Sigma' = A diag(s^2) A^T + 0.3 I
    float a0[3], a1[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      a0[k] = m0[0] * R[k] + m0[1] * R[3 + k] + m0[2] * R[6 + k];
      a1[k] = m1[0] * R[k] + m1[1] * R[3 + k] + m1[2] * R[6 + k];
    }
    float sa = kLowPass, sb = 0.f, sc = kLowPass;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      sa += a0[k] * a0[k] * ss[k];
      sb += a0[k] * a1[k] * ss[k];
      sc += a1[k] * a1[k] * ss[k];
    }
    const float det = sa * sc - sb * sb;
    if (det > 0.f) {
      const float idet = 1.f / det;
      const float cull = cover_limit(sa, sc, idet, u, v, 2.f * logf(255.f * sig));
      a.splat[i].a = make_float4(u, v, sc * idet, 2.f * (-sb * idet));
      a.splat[i].b = make_float4(sa * idet, sig, cull, 0.f);
      // every pixel centre with alpha >= 1/255 lies within lambda_max * 2 ln(255 sigma)
      // of the mean; one pixel of slack for the FP32 evaluation
      const float half = 0.5f * (sa + sc);
      const float lmax = half + sqrtf(fmaxf(0.25f * (sa - sc) * (sa - sc) + sb * sb, 0.f));
      const float rad = sqrtf(lmax * 2.f * logf(255.f * sig)) + 1.f;
      // tile bounds clamped to [-1, tiles] before the integer conversion (u, v or rad may be huge)
      const float ftx = float(cam.tx), fty = float(cam.ty);
      const int x0 = max(0, int(fminf(fmaxf(floorf((u - rad - 0.5f) / kTile), -1.f), ftx)));
      const int x1 = min(cam.tx - 1, int(fminf(fmaxf(floorf((u + rad - 0.5f) / kTile), -1.f), ftx)));
      const int y0 = max(0, int(fminf(fmaxf(floorf((v - rad - 0.5f) / kTile), -1.f), fty)));
      const int y1 = min(cam.ty - 1, int(fminf(fmaxf(floorf((v + rad - 0.5f) / kTile), -1.f), fty)));
      if (x0 <= x1 && y0 <= y1 && isfinite(u) && isfinite(v) && isfinite(rad)) {
        *square = uint32_t((x1 - x0 + 1) * (y1 - y0 + 1));
        const CoverRows rows = cover_rows(u, v, sa, sb, sc, det, cull);
        for (int ty = y0; ty <= y1; ++ty) {
          int c0, c1;
          if (!cover_row(rows, ty, x0, x1, &c0, &c1)) continue;
          count += uint32_t(c1 - c0 + 1);
          count_tiles(counts, (uint32_t(ty) << a.td.x_bits) + uint32_t(c0), (uint32_t(ty) << a.td.x_bits) + uint32_t(c1),
                      a.td);
        }
        if (count) {
          a.rows[i] = rows;
          a.rect[i] = make_uint2(uint32_t(x0) | uint32_t(x1) << 16, uint32_t(y0) | uint32_t(y1) << 16);
          a.reach[i] = count;
        }
      }
    }
  }
  // depth sort key: the bits of a positive float order like its value
  *key = count ? __float_as_uint(pz) : sort::kNone;
  return count;
}

// Projection of every primitive and, beside it, all the counts that the sorts start from, which
// would otherwise take a launch over the keys for each pass (1e6 primitives, 1.4e7 pairs of squares: 58 us
// here, of them 16 us the projection; as launches of their own the counts took 98 us). Bound: the atomics on the
// block's shared counts. The grid is a few blocks per SM, so that those go to global memory once for many
// primitives.
__global__ void __launch_bounds__(kBlock) project_kernel(const ProjectArgs a) {
  __shared__ Counts counts;
  __shared__ unsigned long long s_pairs;
  __shared__ uint32_t s_drawn, warp_tot[kBlock / 32];
  const int t = threadIdx.x, lane = t & 31;
  for (int j = 0; j < kDepthPasses; ++j) counts.depth[j][t] = 0;
  for (int j = 0; j < kMaxTilePasses; ++j) {
    counts.tile[j][t] = 0;
    if (t == 0) counts.tile[j][sort::kBins] = 0;
  }
  if (t == 0) {
    s_pairs = 0;
    s_drawn = 0;
  }
  __syncthreads();
  unsigned long long pairs = 0;
  uint32_t drawn = 0;
  for (int64_t base = int64_t(blockIdx.x) * kBlock; base < a.n; base += int64_t(gridDim.x) * kBlock) {
    const int64_t i = base + t;
    uint32_t square = 0, key = sort::kNone;
    if (i < a.n) {
      if (project_one(a, i, counts, &square, &key)) ++drawn;
      a.dkey[i] = key;
    }
    pairs += square;
    __syncwarp();
    // nearby depths share their upper digits: those are merged within the warp
    const bool ok = key != sort::kNone;
    if (ok) {
      atomicAdd(&counts.depth[0][key & 255u], 1u);
      atomicAdd(&counts.depth[1][(key >> 8) & 255u], 1u);
    }
    count_merged(counts.depth[2], ok ? (key >> 16) & 255u : 256u, lane);
    count_merged(counts.depth[3], ok ? key >> 24 : 256u, lane);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    pairs += __shfl_xor_sync(0xffffffffu, pairs, o);
    drawn += __shfl_xor_sync(0xffffffffu, drawn, o);
  }
  if (lane == 0) {
    atomicAdd(&s_pairs, pairs);
    atomicAdd(&s_drawn, drawn);
  }
  __syncthreads();
  chain_next();
  uint32_t unused;
  const uint32_t d = counts.tile[0][t];
  const uint32_t low = sort::block_scan<kBlock>(d, warp_tot, &unused) + d;
  if (t < (1 << a.td.bits[0]) && low) atomicAdd(&a.hdr->tile_hist[0][t], low);
  for (int j = 1; j < a.td.passes; ++j)
    if (counts.tile[j][t]) atomicAdd(&a.hdr->tile_hist[j][t], counts.tile[j][t]);
  for (int j = 0; j < kDepthPasses; ++j)
    if (counts.depth[j][t]) atomicAdd(&a.hdr->depth_hist[j][t], counts.depth[j][t]);
  if (t == 0) {
    if (s_pairs) atomicAdd(&a.hdr->pairs64, s_pairs);
    if (s_drawn) atomicAdd(&a.hdr->drawn, s_drawn);
    __threadfence();
    if (atomicAdd(&a.hdr->projected, 1u) == gridDim.x - 1) {  // the last block tells the host
      volatile HostTotal* host = a.host;
      host->pairs = atomicAdd(&a.hdr->pairs64, 0ull);
      __threadfence_system();
      host->call = a.call;
    }
  }
}

// ---------------------------------------------------------------------------
// Sorts
// ---------------------------------------------------------------------------

// The block's ticket and the exclusive sum of the pass's digit counts.
template <int THREADS, int ITEMS>
__device__ __forceinline__ uint32_t take_ticket(sort::Block<THREADS, ITEMS>& s, const sort::Pass& ps, uint32_t* digit_base) {
  const int t = threadIdx.x;
  chain_wait();
  if (t == 0) {
    s.ticket = atomicAdd(ps.ticket, 1u);
    s.stop = *ps.failed;
  }
  uint32_t unused;
  *digit_base = sort::block_scan<THREADS>(t < (1 << ps.bits) ? ps.hist[t] : 0u, s.warp_tot, &unused);
  return s.ticket;
}

// One pass of the depth sort over *count entries (n in the first, which drops what is not
// drawn and whose values are the places). The last needs no keys.
template <int THREADS, int ITEMS, bool FIRST, bool LAST>
__global__ void __launch_bounds__(THREADS, THREADS > 256 ? 2 : 4) depth_pass_kernel(sort::Pass ps, const uint32_t* __restrict__ kin,
                                                            const uint32_t* __restrict__ vin,
                                                            uint32_t* __restrict__ kout, uint32_t* __restrict__ vout,
                                                            uint32_t n, const uint32_t* __restrict__ drawn) {
  extern __shared__ __align__(16) unsigned char sort_smem[];
  auto& s = *reinterpret_cast<sort::Block<THREADS, ITEMS>*>(sort_smem);
  uint32_t digit_base;
  const uint32_t block = take_ticket(s, ps, &digit_base);
  const uint32_t m = FIRST ? n : *drawn;
  if (uint64_t(block) * (THREADS * ITEMS) >= m || s.stop) return;
  const uint32_t at = block * (THREADS * ITEMS) + (threadIdx.x >> 5) * (32 * ITEMS) + (threadIdx.x & 31);
  uint32_t key[ITEMS], val[ITEMS];
#pragma unroll
  for (int i = 0; i < ITEMS; ++i) {
    const uint32_t j = at + 32 * i;
    key[i] = j < m ? kin[j] : sort::kNone;
    val[i] = FIRST ? j : (j < m ? vin[j] : 0u);
  }
  const int cnt = sort::sort_block<THREADS, ITEMS, LAST>(s, ps, block, digit_base, key, val);
  chain_next();
  const uint32_t mask = (1u << ps.bits) - 1u;
  for (int p = threadIdx.x; p < cnt; p += THREADS) {
    const uint32_t k = s.key[p];
    const uint32_t dst = s.base[(k >> ps.shift) & mask] + uint32_t(p);
    if (!LAST) kout[dst] = k;
    vout[dst] = s.val[p];
  }
}

// Exclusive scan, in depth order, of the tiles each drawn primitive reaches: its first pair. Notes
// for every kStartGrain-th pair the primitive it belongs to, and the total; clears the pair passes'
// states (as far as these pairs need them) on the way. It runs before the host has compared the
// squares' pairs with the capacity: where they exceed it, nothing sized by the capacity is written.
__global__ void __launch_bounds__(kBlock) offsets_kernel(Header* hdr, uint32_t* ticket, int* err,
                                                         unsigned long long cap,
                                                         ulonglong2* __restrict__ pair_states,
                                                         unsigned long long* __restrict__ states,
                                                         const uint32_t* __restrict__ order,
                                                         const uint32_t* __restrict__ reach,
                                                         uint32_t* __restrict__ offsets, uint32_t* __restrict__ starts) {
  __shared__ uint32_t warp_tot[kBlock / 32], s_ticket, s_stop, s_before;
  __shared__ int s_ok;
  constexpr uint32_t kChunk = kBlock * kScanItems;
  const int t = threadIdx.x;
  chain_wait();
  // the pair passes' states start at zero
  const unsigned long long squares = hdr->pairs64;
  if (squares <= cap) {
    const int64_t words = sort_blocks(int64_t(squares), kLargePairs) * sort::kBins / 2;
    for (int64_t i = int64_t(blockIdx.x) * kBlock + t; i < words; i += int64_t(gridDim.x) * kBlock)
      pair_states[i] = make_ulonglong2(0ull, 0ull);
  }
  if (t == 0) {
    s_ticket = atomicAdd(ticket, 1u);
    s_stop = hdr->failed;
  }
  __syncthreads();
  const uint32_t block = s_ticket, n = hdr->drawn;
  if (uint64_t(block) * kChunk >= n || s_stop) return;
  const uint32_t k0 = block * kChunk + uint32_t(t) * kScanItems;
  static_assert(kScanItems % 4 == 0, "order and offsets move four at a time");
  uint32_t c[kScanItems], sum = 0;
#pragma unroll
  for (int i = 0; i < kScanItems; i += 4) {
    // past n the order's buffer holds stale entries (it has room for whole groups of four)
    const uint4 id = k0 + i < n ? *reinterpret_cast<const uint4*>(order + k0 + i) : make_uint4(0u, 0u, 0u, 0u);
    c[i] = k0 + i < n ? reach[id.x] : 0u;
    c[i + 1] = k0 + i + 1 < n ? reach[id.y] : 0u;
    c[i + 2] = k0 + i + 2 < n ? reach[id.z] : 0u;
    c[i + 3] = k0 + i + 3 < n ? reach[id.w] : 0u;
  }
#pragma unroll
  for (int i = 0; i < kScanItems; ++i) sum += c[i];
  uint32_t total;
  uint32_t run = sort::block_scan<kBlock>(sum, warp_tot, &total);
  constexpr uint32_t kTag = 1;
  if (t < 32) {
    if (t == 0) sort::st_state(states + block, (block == 0 ? sort::kAll : sort::kOwn) | sort::tag_bits(kTag) | total);
    unsigned long long before = 0;
    const bool ok = block == 0 || sort::look_back_warp(states, block, kTag, kWaitLimit, err, &before);
    if (t == 0) {
      if (block > 0)
        sort::st_state(states + block,
                       (ok ? sort::kAll : sort::kGone) | sort::tag_bits(kTag) | ((before + total) & sort::kCount));
      s_before = uint32_t(before);
      s_ok = ok;
      if (!ok) hdr->failed = 1;
      if (uint64_t(block + 1) * kChunk >= n) hdr->pairs = uint32_t(before) + total;
    }
  }
  __syncthreads();
  if (!s_ok) return;
  chain_next();
  run += s_before;
  uint32_t first[kScanItems];
#pragma unroll
  for (int i = 0; i < kScanItems; ++i) {
    first[i] = run;
    if (k0 + i < n && squares <= cap) {  // a forward that will be refused has no room in starts
      for (uint64_t b = (uint64_t(run) + kStartGrain - 1) / kStartGrain; b * kStartGrain < uint64_t(run) + c[i]; ++b)
        starts[b] = k0 + i;
    }
    run += c[i];
  }
#pragma unroll
  for (int i = 0; i < kScanItems; i += 4)
    if (k0 + i < n)
      *reinterpret_cast<uint4*>(offsets + k0 + i) = make_uint4(first[i], first[i + 1], first[i + 2], first[i + 3]);
}

// Writes a sorted block of pairs; the last pass also takes the ends of the tiles' runs into the
// ranges (x: the largest complement of a place, so that zero means none; y: the largest place + 1).
template <int THREADS, int ITEMS, bool LAST>
__device__ __forceinline__ void write_pairs(const sort::Block<THREADS, ITEMS>& s, const sort::Pass& ps, int cnt,
                                            uint32_t* __restrict__ kout, uint32_t* __restrict__ vout, uint2* ranges,
                                            int x_bits, int tiles_x) {
  const uint32_t mask = (1u << ps.bits) - 1u;
  for (int p = threadIdx.x; p < cnt; p += THREADS) {
    const uint32_t k = s.key[p];
    const uint32_t dst = s.base[(k >> ps.shift) & mask] + uint32_t(p);
    vout[dst] = s.val[p];
    if (LAST) {
      uint2* r = ranges + (k >> x_bits) * uint32_t(tiles_x) + (k & ((1u << x_bits) - 1u));
      if (p == 0 || s.key[p - 1] != k) atomicMax(&r->x, ~dst);
      if (p == cnt - 1 || s.key[p + 1] != k) atomicMax(&r->y, dst + 1u);
    } else {
      kout[dst] = k;
    }
  }
}

struct ListArgs {
  Header* hdr;
  const uint32_t* order;
  const uint32_t* offsets;
  const uint32_t* starts;
  const uint2* rect;
  const uint32_t* reach;
  const CoverRows* rows;
  int x_bits;   // of a tile's key
  int tiles_x;
};

// First pass of the pair sort (1e6 primitives at 1080p: 111 us; issue 39 % active, the leading stalls
// barriers, loads of the primitives' rows and shared-memory traffic). A block's pairs are places [base, base + THREADS ITEMS) of the depth
// order's list: it finds the primitives that hold them in `starts` and writes their tiles into
// shared memory itself, so the list never goes through memory unsorted. A thread lists a
// primitive of up to kAlone tiles alone; a warp shares the rows of a larger one.
template <int THREADS, int ITEMS, bool LAST>
__global__ void __launch_bounds__(THREADS, THREADS > 256 ? 2 : 4) list_pass_kernel(ListArgs a, sort::Pass ps, uint32_t* __restrict__ kout,
                                                           uint32_t* __restrict__ vout, uint2* ranges) {
  constexpr uint32_t kAlone = 64;
  constexpr uint32_t kPer = THREADS * ITEMS;
  extern __shared__ __align__(16) unsigned char sort_smem[];
  auto& s = *reinterpret_cast<sort::Block<THREADS, ITEMS>*>(sort_smem);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  uint32_t digit_base;
  const uint32_t block = take_ticket(s, ps, &digit_base);
  const uint32_t pairs = a.hdr->pairs, drawn = a.hdr->drawn;
  if (uint64_t(block) * kPer >= pairs || s.stop) return;
  const uint32_t base = block * kPer;
  const uint32_t size = min(kPer, pairs - base);
  // o: the primitive's first place less base; negative (by less than its tiles, at most 2^20)
  // where it starts before the block
  for (uint32_t k = a.starts[block * (kPer / kStartGrain)] + threadIdx.x;; k += THREADS) {
    const int64_t far = k < drawn ? int64_t(a.offsets[k]) - int64_t(base) : int64_t(size);
    const int first = int(min(far, int64_t(size)));
    int o = first;
    const bool act = o < int(size);
    if (!__any_sync(0xffffffffu, act)) break;  // the offsets only grow
    uint32_t id = 0, reach = 0;
    uint2 rc = make_uint2(0, 0);
    if (act) {
      id = a.order[k];
      rc = a.rect[id];
      reach = a.reach[id];
    }
    if (act && reach <= kAlone) {
      const CoverRows rows = a.rows[id];
      const int y1 = int(rc.y >> 16);
      for (int ty = int(rc.y & 0xffffu); ty <= y1; ++ty) {
        int c0, c1;
        if (!cover_row(rows, ty, int(rc.x & 0xffffu), int(rc.x >> 16), &c0, &c1)) continue;
        for (int tx = c0; tx <= c1; ++tx, ++o)
          if (uint32_t(o) < size) {
            s.key[o] = (uint32_t(ty) << a.x_bits) + uint32_t(tx);
            s.val[o] = id;
          }
      }
    }
    uint32_t big = __ballot_sync(0xffffffffu, act && reach > kAlone);
    while (big) {
      const int src = __ffs(int(big)) - 1;
      big &= big - 1;
      int run = __shfl_sync(0xffffffffu, first, src);
      const uint32_t bid = __shfl_sync(0xffffffffu, id, src);
      const uint2 br = a.rect[bid];
      const CoverRows rows = a.rows[bid];
      const int y1 = int(br.y >> 16);
      for (int r0 = int(br.y & 0xffffu); r0 <= y1 && run < int(size); r0 += 32) {
        int c0 = 0, c1 = -1;
        const int ty = r0 + lane;
        if (ty > y1 || !cover_row(rows, ty, int(br.x & 0xffffu), int(br.x >> 16), &c0, &c1)) c1 = c0 - 1;
        const uint32_t len = uint32_t(c1 - c0 + 1);
        uint32_t inc = len;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
          const uint32_t y = __shfl_up_sync(0xffffffffu, inc, d);
          if (lane >= d) inc += y;
        }
        const int at = run + int(inc - len);
        const int to = min(int(len), int(size) - at);
        for (int j = max(0, -at); j < to; ++j) {
          s.key[at + j] = (uint32_t(ty) << a.x_bits) + uint32_t(c0 + j);
          s.val[at + j] = bid;
        }
        run += int(__shfl_sync(0xffffffffu, inc, 31));
      }
    }
  }
  __syncthreads();
  uint32_t key[ITEMS], val[ITEMS];
#pragma unroll
  for (int i = 0; i < ITEMS; ++i) {
    const uint32_t p = uint32_t(warp * 32 * ITEMS + 32 * i + lane);
    key[i] = p < size ? s.key[p] : sort::kNone;
    val[i] = p < size ? s.val[p] : 0u;
  }
  const int cnt = sort::sort_block<THREADS, ITEMS, true>(s, ps, block, digit_base, key, val);
  chain_next();
  write_pairs<THREADS, ITEMS, LAST>(s, ps, cnt, kout, vout, ranges, a.x_bits, a.tiles_x);
}

// A later pass of the pair sort.
template <int THREADS, int ITEMS, bool LAST>
__global__ void __launch_bounds__(THREADS, THREADS > 256 ? 2 : 4) pair_pass_kernel(Header* hdr, sort::Pass ps,
                                                           const uint32_t* __restrict__ kin,
                                                           const uint32_t* __restrict__ vin,
                                                           uint32_t* __restrict__ kout, uint32_t* __restrict__ vout,
                                                           uint2* ranges, int x_bits, int tiles_x) {
  extern __shared__ __align__(16) unsigned char sort_smem[];
  auto& s = *reinterpret_cast<sort::Block<THREADS, ITEMS>*>(sort_smem);
  uint32_t digit_base;
  const uint32_t block = take_ticket(s, ps, &digit_base), m = hdr->pairs;
  if (uint64_t(block) * (THREADS * ITEMS) >= m || s.stop) return;
  const uint32_t at = block * (THREADS * ITEMS) + (threadIdx.x >> 5) * (32 * ITEMS) + (threadIdx.x & 31);
  uint32_t key[ITEMS], val[ITEMS];
#pragma unroll
  for (int i = 0; i < ITEMS; ++i) {
    const uint32_t j = at + 32 * i;
    key[i] = j < m ? kin[j] : sort::kNone;
    val[i] = j < m ? vin[j] : 0u;
  }
  const int cnt = sort::sort_block<THREADS, ITEMS, false>(s, ps, block, digit_base, key, val);
  chain_next();
  write_pairs<THREADS, ITEMS, LAST>(s, ps, cnt, kout, vout, ranges, x_bits, tiles_x);
}

// The list of a tile; empty where a sort gave up.
__device__ __forceinline__ TileList list_of(const Header* hdr, const uint2* __restrict__ ranges, int tile) {
  const uint2 r = ranges[tile];
  return hdr->failed ? TileList{0u, 0u} : tile_list(r.x, r.y);
}

// ---------------------------------------------------------------------------
// Tile rendering
// ---------------------------------------------------------------------------

// Bound: issue (78 % of the slots in both passes at 1e6 primitives and 1920 x 1080, 258 us forward and 405 us
// backward; FMA pipe 49 and 42 % busy, DRAM idle at 2 %). Most primitives whose footprint square meets a tile
// miss most of its pixels: masks per 8 x 8 or 8 x 4 sub-tile cost one thread about 40 operations per
// (tile, primitive) and save the warps the visits. Two pixels per lane share the staged reads, the terms in
// x and, backward, the shuffles; a tile adds each of its sums once.
//
// Pixels of a tile among its warps. PX = 2: four warps, one 8 x 8 quadrant each, a lane
// holding pixels (x, y) and (x, y + 4); PX = 1: eight warps of 8 x 4 pixels, one per lane.
template <int PX>
struct TileShape {
  static constexpr int NT = kTilePixels / PX;   // threads, and primitives per staged batch
  static constexpr int W = NT / 32;             // warps = sub-tiles
  static constexpr int H = 4 * PX;              // sub-tile height (width 8)
  static constexpr int WORDS = NT / 32;         // mask words per sub-tile and batch
};

// Staged primitives of a batch. PX = 2: every operand of the two pixels' packed arithmetic twice.
template <int PX>
struct Stage {
  static constexpr int NT = TileShape<PX>::NT;
  float4 mean[NT];                                        // PX 2: -x, -x, -y, -y; PX 1: x, y, A, 2B
  float4 form[NT];                                        // PX 2: A, A, 2B, 2B;   PX 1: C, sigma, 0, 0
  float4 rest[PX == 2 ? NT : 1];                          // PX 2: C, C, sigma, sigma
  float4 colour[NT];                                      // red, green, blue, sigma
  uint32_t mask[TileShape<PX>::W][TileShape<PX>::WORDS];  // primitives that can reach each sub-tile
};

// Which sub-tiles (bit w) of the tile at pixel (x0, y0) the primitive's ellipse can reach.
template <int PX>
__device__ __forceinline__ uint32_t reach_mask(const Splat& p, float x0, float y0) {
  using TS = TileShape<PX>;
  const float cull = p.b.z;
  if (!(cull < INFINITY)) return (1u << TS::W) - 1u;
  const CoverSlopes r = cover_slopes(p.a.z, p.a.w, p.b.x);
  uint32_t m = 0;
#pragma unroll
  for (int w = 0; w < TS::W; ++w) {
    const float fx = x0 + float(w & 1) * 8.f + 0.5f, fy = y0 + float(w >> 1) * float(TS::H) + 0.5f;
    if (cover_box(p.a.z, p.a.w, p.b.x, r, cull, fx - p.a.x, (fx + 7.f) - p.a.x, fy - p.a.y,
                  (fy + float(TS::H - 1)) - p.a.y))
      m |= 1u << w;
  }
  return m;
}

// Stages primitive list[j] (where `has`) in slot threadIdx.x and the batch's masks. Each warp
// stages 32 slots and turns their reach masks into one word per sub-tile.
template <int PX>
__device__ __forceinline__ void stage_batch(Stage<PX>& st, const uint32_t* __restrict__ list, bool has, uint32_t j, float x0,
                                            float y0, const Splat* __restrict__ splat,
                                            const float* __restrict__ colours, uint32_t* id_out) {
  using TS = TileShape<PX>;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  uint32_t m = 0;
  if (has) {
    const uint32_t id = list[j];
    if (id_out) *id_out = id;
    Splat p;
    p.a = splat[id].a;
    p.b = splat[id].b;
    const float* c = colours + 3 * int64_t(id);
    const int t = threadIdx.x;
    if constexpr (PX == 2) {
      st.mean[t] = make_float4(-p.a.x, -p.a.x, -p.a.y, -p.a.y);
      st.form[t] = make_float4(p.a.z, p.a.z, p.a.w, p.a.w);
      st.rest[t] = make_float4(p.b.x, p.b.x, p.b.y, p.b.y);
    } else {
      st.mean[t] = p.a;
      st.form[t] = make_float4(p.b.x, p.b.y, 0.f, 0.f);
    }
    st.colour[t] = make_float4(c[0], c[1], c[2], p.b.y);
    m = reach_mask<PX>(p, x0, y0);
  }
#pragma unroll
  for (int w = 0; w < TS::W; ++w) {
    const uint32_t word = __ballot_sync(0xffffffffu, (m >> w) & 1u);
    if (lane == w) st.mask[w][warp] = word;
  }
}

// alpha of staged primitive k at the lane's pixels; 0 when below 1/255. Every operation is
// explicitly rounded so that the forward and the backward kernels take the same decisions on
// the same inputs. Two pixels go through packed FP32x2 operations, each component rounded as the
// scalar one, so both layouts give the same bits (1080p, 1e6 primitives: forward 261 us, with
// scalar operations 271 us, backward 415 and 432 us; the operands are staged twice to be had without moves).
template <int PX>
__device__ __forceinline__ void pixel_alpha(const Stage<PX>& st, int k, float px, const float* py, float* alpha,
                                            float* rho) {
  if constexpr (PX == 2) {
    const float4 m = st.mean[k], f = st.form[k], r = st.rest[k];
    const float2 dx = __fadd2_rn(make_float2(px, px), make_float2(m.x, m.y));
    const float2 dy = __fadd2_rn(make_float2(py[0], py[1]), make_float2(m.z, m.w));
    const float2 adx = __fmul2_rn(make_float2(f.x, f.y), dx), bdx = __fmul2_rn(make_float2(f.z, f.w), dx);
    const float2 cdy = __fmul2_rn(__fmul2_rn(make_float2(r.x, r.y), dy), dy);
    const float2 q = __ffma2_rn(adx, dx, __ffma2_rn(bdx, dy, cdy));
    const float2 e = __fmul2_rn(q, make_float2(kExpScale, kExpScale));
    rho[0] = ex2a(e.x);
    rho[1] = ex2a(e.y);
    const float2 al = __fmul2_rn(make_float2(r.z, r.w), make_float2(rho[0], rho[1]));
    alpha[0] = fminf(kAlphaMax, al.x);
    alpha[1] = fminf(kAlphaMax, al.y);
  } else {
    const float4 m = st.mean[k], f = st.form[k];
    const float dx = __fsub_rn(px, m.x), dy = __fsub_rn(py[0], m.y);
    const float q = __fmaf_rn(__fmul_rn(m.z, dx), dx,
                              __fmaf_rn(__fmul_rn(m.w, dx), dy, __fmul_rn(__fmul_rn(f.x, dy), dy)));
    rho[0] = ex2a(__fmul_rn(q, kExpScale));
    alpha[0] = fminf(kAlphaMax, __fmul_rn(f.y, rho[0]));
  }
#pragma unroll
  for (int p = 0; p < PX; ++p) alpha[p] = alpha[p] >= kAlphaMin ? alpha[p] : 0.f;
}

template <int PX>
__global__ void __launch_bounds__(TileShape<PX>::NT) render_fwd_kernel(
    Cam cam, const Header* __restrict__ hdr, const uint2* __restrict__ ranges, const uint32_t* __restrict__ vals,
    const Splat* __restrict__ splat, const float* __restrict__ colours, float* __restrict__ image, float* __restrict__ final_t,
    uint32_t* __restrict__ ncontrib) {
  using TS = TileShape<PX>;
  __shared__ Stage<PX> st;
  chain_wait();
  const int tile = blockIdx.x;
  const int tx = tile % cam.tx, ty = tile / cam.tx;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int pxi = tx * kTile + (warp & 1) * 8 + (lane & 7);
  const int pyi = ty * kTile + (warp >> 1) * TS::H + (lane >> 3);
  const float px = float(pxi) + 0.5f;
  const TileList list = list_of(hdr, ranges, tile);
  float py[PX], T[PX], c0[PX], c1[PX], c2[PX];
  uint32_t last[PX];
  bool done[PX], inside[PX];
#pragma unroll
  for (int p = 0; p < PX; ++p) {
    py[p] = float(pyi + 4 * p) + 0.5f;
    T[p] = 1.f;
    c0[p] = c1[p] = c2[p] = 0.f;
    last[p] = 0;
    inside[p] = pxi < cam.w && pyi + 4 * p < cam.h;
    done[p] = !inside[p];
  }
  bool live = true;  // warp-uniform: some pixel of the warp has not stopped
  for (ListWalk b(list); b.left > 0; b.next(TS::NT)) {
    bool all = true;
#pragma unroll
    for (int p = 0; p < PX; ++p) all = all && done[p];
    live = !__all_sync(0xffffffffu, all);
    if (!__syncthreads_or(live)) break;
    stage_batch<PX>(st, vals, threadIdx.x < b.left, b.place + threadIdx.x, float(tx * kTile), float(ty * kTile), splat,
                    colours, nullptr);
    __syncthreads();
    for (int q = 0; live && q < TS::WORDS; ++q) {
      uint32_t m = st.mask[warp][q];
      while (m) {
        const int k = 32 * q + __ffs(int(m)) - 1;
        m &= m - 1;
        float al[PX], rho[PX];
        pixel_alpha<PX>(st, k, px, py, al, rho);
        const float4 col = st.colour[k];
#pragma unroll
        for (int p = 0; p < PX; ++p) {
          if (al[p] != 0.f && !done[p]) {
            const float test = T[p] * (1.f - al[p]);
            if (test < kTMin) {
              done[p] = true;
            } else {
              const float w = al[p] * T[p];
              c0[p] = fmaf(col.x, w, c0[p]);
              c1[p] = fmaf(col.y, w, c1[p]);
              c2[p] = fmaf(col.z, w, c2[p]);
              T[p] = test;
              last[p] = b.place - list.begin + uint32_t(k) + 1;
            }
          }
        }
      }
      all = true;
#pragma unroll
      for (int p = 0; p < PX; ++p) all = all && done[p];
      live = !__all_sync(0xffffffffu, all);
    }
  }
#pragma unroll
  for (int p = 0; p < PX; ++p) {
    if (!inside[p]) continue;
    const int64_t at = int64_t(pyi + 4 * p) * cam.w + pxi;
    image[3 * at] = c0[p];
    image[3 * at + 1] = c1[p];
    image[3 * at + 2] = c2[p];
    final_t[at] = T[p];
    ncontrib[at] = last[p];
  }
}

template <int PX>
__global__ void __launch_bounds__(TileShape<PX>::NT) render_bwd_kernel(
    Cam cam, const Header* __restrict__ hdr, const uint2* __restrict__ ranges, const uint32_t* __restrict__ vals,
    const Splat* __restrict__ splat, const float* __restrict__ colours, const float* __restrict__ final_t, const uint32_t* __restrict__ ncontrib,
    const float* __restrict__ g_image, float* __restrict__ g_colours, float* __restrict__ g_opacity) {
  using TS = TileShape<PX>;
  __shared__ Stage<PX> st;
  __shared__ float4 s_grad[TS::W][TS::NT];  // each warp's sums for the staged primitives
  __shared__ uint32_t s_last;
  const int tile = blockIdx.x;
  const int tx = tile % cam.tx, ty = tile / cam.tx;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int pxi = tx * kTile + (warp & 1) * 8 + (lane & 7);
  const int pyi = ty * kTile + (warp >> 1) * TS::H + (lane >> 3);
  const float px = float(pxi) + 0.5f;
  const uint32_t* __restrict__ list = vals + list_of(hdr, ranges, tile).begin;
  float py[PX], T[PX], g0[PX], g1[PX], g2[PX];
  float after[PX];  // sum over later contributions of (c . g) alpha T
  uint32_t last[PX];
  uint32_t most = 0;
#pragma unroll
  for (int p = 0; p < PX; ++p) {
    const bool inside = pxi < cam.w && pyi + 4 * p < cam.h;
    const int64_t at = int64_t(pyi + 4 * p) * cam.w + pxi;
    py[p] = float(pyi + 4 * p) + 0.5f;
    T[p] = inside ? final_t[at] : 1.f;
    last[p] = inside ? ncontrib[at] : 0u;
    g0[p] = inside ? g_image[3 * at] : 0.f;
    g1[p] = inside ? g_image[3 * at + 1] : 0.f;
    g2[p] = inside ? g_image[3 * at + 2] : 0.f;
    after[p] = 0.f;
    most = max(most, last[p]);
  }
  // batches from the back of the range, starting at the block's furthest last
  // contribution (entries behind every pixel's stop point contribute nothing)
  if (threadIdx.x == 0) s_last = 0;
  __syncthreads();
  most = __reduce_max_sync(0xffffffffu, most);  // of the warp's pixels
  if (lane == 0) atomicMax(&s_last, most);
  __syncthreads();
  const uint32_t n = s_last;
  for (uint32_t seen = 0; seen < n; seen += TS::NT) {
    const uint32_t hi = n - seen;                            // exclusive end (relative)
    const uint32_t lo = hi > uint32_t(TS::NT) ? hi - TS::NT : 0u;
    uint32_t id = 0;
    stage_batch<PX>(st, list, lo + threadIdx.x < hi, lo + threadIdx.x, float(tx * kTile), float(ty * kTile), splat,
                    colours, &id);
#pragma unroll
    for (int w = 0; w < TS::W; ++w) s_grad[w][threadIdx.x] = make_float4(0.f, 0.f, 0.f, 0.f);
    __syncthreads();
    for (int q = TS::WORDS - 1; q >= 0; --q) {
      uint32_t m = st.mask[warp][q];
      const uint32_t first = lo + 32u * uint32_t(q);         // list position of the word's first entry
      if (first >= most) m = 0;
      else if (most - first < 32u) m &= (1u << (most - first)) - 1u;
      while (m) {
        const int bit = 31 - __clz(int(m));
        m ^= 1u << bit;
        const int k = 32 * q + bit;
        const uint32_t pos = lo + uint32_t(k);               // position in the tile's list
        float al[PX], rho[PX];
        pixel_alpha<PX>(st, k, px, py, al, rho);
        bool any = false;
#pragma unroll
        for (int p = 0; p < PX; ++p) {
          if (pos >= last[p]) al[p] = 0.f;
          any = any || al[p] > 0.f;
        }
        if (!__any_sync(0xffffffffu, any)) continue;
        float gc0 = 0.f, gc1 = 0.f, gc2 = 0.f, go = 0.f;
        const float4 col = st.colour[k];
#pragma unroll
        for (int p = 0; p < PX; ++p) {
          if (al[p] > 0.f) {
            // 1/(1 - alpha), 1 - alpha in [0.01, 1]: the approximation and one Newton step, against 64
            // bits no further off than the division (g_opacity 1.01e-6 either way at 1080p, without the
            // pixels whose stop differs) and a third of its instructions (1080p: 432 us, divided 489 us)
            const float om = 1.f - al[p], r0 = rcpa(om);
            const float inv = fmaf(r0, fmaf(-om, r0, 1.f), r0);
            const float Tb = T[p] * inv;  // transmittance in front of this contribution
            const float w = al[p] * Tb;
            gc0 = fmaf(w, g0[p], gc0);
            gc1 = fmaf(w, g1[p], gc1);
            gc2 = fmaf(w, g2[p], gc2);
            const float cg = fmaf(g2[p], col.z, fmaf(g1[p], col.y, g0[p] * col.x));
            if (col.w * rho[p] < kAlphaMax) go = fmaf(cg * Tb - after[p] * inv, rho[p], go);
            after[p] = fmaf(cg, w, after[p]);
            T[p] = Tb;
          }
        }
        // four sums over the warp in six shuffles: halves exchange two values, then
        // quarters one, then a plain butterfly; lane 8 q (q = 0..3) ends with sum q
        const bool hi16 = (lane & 16) != 0, hi8 = (lane & 8) != 0;
        float k0 = hi16 ? gc2 : gc0, k1 = hi16 ? go : gc1;
        const float s0 = hi16 ? gc0 : gc2, s1 = hi16 ? gc1 : go;
        k0 += __shfl_xor_sync(0xffffffffu, s0, 16);
        k1 += __shfl_xor_sync(0xffffffffu, s1, 16);
        float v = hi8 ? k1 : k0;
        v += __shfl_xor_sync(0xffffffffu, hi8 ? k0 : k1, 8);
        v += __shfl_xor_sync(0xffffffffu, v, 4);
        v += __shfl_xor_sync(0xffffffffu, v, 2);
        v += __shfl_xor_sync(0xffffffffu, v, 1);
        if ((lane & 7) == 0) reinterpret_cast<float*>(&s_grad[warp][k])[lane >> 3] = v;
      }
    }
    __syncthreads();
    // thread k adds the warps' sums of staged primitive k to its gradients
    if (threadIdx.x < hi - lo) {
      float4 g = s_grad[0][threadIdx.x];
#pragma unroll
      for (int w = 1; w < TS::W; ++w) {
        const float4 h = s_grad[w][threadIdx.x];
        g.x += h.x; g.y += h.y; g.z += h.z; g.w += h.w;
      }
      if (g.x != 0.f) atomicAdd(g_colours + 3 * int64_t(id), g.x);
      if (g.y != 0.f) atomicAdd(g_colours + 3 * int64_t(id) + 1, g.y);
      if (g.z != 0.f) atomicAdd(g_colours + 3 * int64_t(id) + 2, g.z);
      if (g.w != 0.f) atomicAdd(g_opacity + id, g.w);
    }
    __syncthreads();
  }
}

// One pixel per lane gives each tile twice the warps, which hides the chain through a pixel's
// list where the image has few tiles. Backward alone, one / two pixels per lane: 60 tiles (1e5
// primitives) 114 / 152 us, 240 tiles 89 / 114, 510 tiles 99 / 109, 920 tiles 116 / 99, 8160 tiles
// 540 / 414: the line at four tiles per SM. Whole forward: 510 tiles 202 / 209, 920 tiles 183 / 195,
// 2040 tiles 237.2 / 236.8 and 167 / 162, 3600 tiles 283 / 270, 8160 tiles 595 / 559: at eight.
inline bool two_pixels(int64_t tiles, int per_sm) { return tiles >= int64_t(per_sm) * sm_count(); }

inline Cam make_cam(const nasg_raster_camera* c) {
  Cam k;
  for (int j = 0; j < 9; ++j) k.r[j] = c->rot[j];
  for (int j = 0; j < 3; ++j) k.c[j] = c->centre[j];
  k.fx = c->fx;
  k.fy = c->fy;
  k.cx = c->cx;
  k.cy = c->cy;
  k.near_z = c->near_z;
  k.w = c->width;
  k.h = c->height;
  k.tx = (c->width + kTile - 1) / kTile;
  k.ty = (c->height + kTile - 1) / kTile;
  return k;
}

inline bool camera_ok(const nasg_raster_camera* c) {
  if (c->width < 1 || c->height < 1 || c->width > 16384 || c->height > 16384) return false;
  if (!(c->fx > 0.f) || !(c->fy > 0.f) || !(c->near_z > 0.f)) return false;
  for (int j = 0; j < 9; ++j)
    if (!std::isfinite(c->rot[j])) return false;
  return std::isfinite(c->cx) && std::isfinite(c->cy) && std::isfinite(c->centre[0]) &&
         std::isfinite(c->centre[1]) && std::isfinite(c->centre[2]);
}

// While it lives, the thread's calls neither fail for nor end a capture that goes on elsewhere (page-locking,
// its release and stream queries are refused during a capture in CUDA's default, global mode).
struct BesideCaptures {
  cudaStreamCaptureMode mode = cudaStreamCaptureModeRelaxed;
  BesideCaptures() { cudaThreadExchangeStreamCaptureMode(&mode); }
  ~BesideCaptures() { cudaThreadExchangeStreamCaptureMode(&mode); }
  BesideCaptures(const BesideCaptures&) = delete;
  BesideCaptures& operator=(const BesideCaptures&) = delete;
};

// The page-locked words of one host thread and the number of its latest call, kept for the thread's
// life (page-locking memory on every call would cost more than the call).
struct HostWords {
  HostTotal* words = nullptr;
  unsigned long long calls = 0;
  ~HostWords() {
    if (!words) return;
    const BesideCaptures beside;
    cudaFreeHost(words);
  }
  bool ready() {
    if (!words) {
      const BesideCaptures beside;
      if (cudaHostAlloc(reinterpret_cast<void**>(&words), sizeof(HostTotal),
                        cudaHostAllocPortable | cudaHostAllocMapped) != cudaSuccess) {
        words = nullptr;
        return false;
      }
      *words = HostTotal{0, 0};
    }
    return true;
  }
};

// For a forward that ends without its image: the pixels' counts are cleared (they are an earlier image's,
// and a backward would take them for places in lists that are not there), and the stream is waited for, so
// that nothing of the call is left running. The caller may then free or reuse the workspace (n_pairs is
// reported so that it can make a larger one), and no late store reaches the thread's words under a later
// call's number.
inline nasg_status give_up(nasg_status why, uint32_t* ncontrib, int64_t pixels, cudaStream_t s) {
  const BesideCaptures beside;
  cudaMemsetAsync(ncontrib, 0, size_t(pixels) * sizeof(uint32_t), s);
  cudaStreamSynchronize(s);
  cudaGetLastError();  // `why` stands; its CUDA error, if it has one, is recorded
  return why;
}

// Waits until the projection of call `call` has left its total (false with the CUDA error recorded
// when the stream fails, is being captured, or finishes without it). The thread polls the word, as the
// runtime's own waits do by default, or waits as the device's scheduling flags ask: yielding between polls,
// or blocked until the stream is done. The flags are read once the first polls have failed.
inline bool wait_total(const HostTotal* words, unsigned long long call, cudaStream_t s, unsigned long long* pairs) {
  const volatile HostTotal* w = words;
  const BesideCaptures beside;
  unsigned schedule = 0;
  for (uint32_t spin = 1;; ++spin) {
    if (w->call == call) break;
    if (schedule == cudaDeviceScheduleYield) std::this_thread::yield();
    if (spin % 1024 != 0) continue;
    if (spin == 1024 && cudaGetDeviceFlags(&schedule) == cudaSuccess) schedule &= cudaDeviceScheduleMask;
    const cudaError_t e = schedule == cudaDeviceScheduleBlockingSync ? cudaStreamSynchronize(s) : cudaStreamQuery(s);
    if (e == cudaErrorNotReady) {
      cudaGetLastError();  // no error
      continue;
    }
    if (e == cudaSuccess && w->call == call) break;
    record_cuda_error(e == cudaSuccess ? cudaErrorUnknown : e);
    cudaGetLastError();
    return false;
  }
  std::atomic_thread_fence(std::memory_order_acquire);
  *pairs = w->pairs;
  return true;
}

// Launches a kernel of the chain: with `chain` it may start while its predecessor runs (see chain_wait).
template <typename... P, typename... A>
nasg_status launch_chained(bool chain, void (*kernel)(P...), unsigned grid, unsigned threads, size_t smem,
                           cudaStream_t s, const A&... args) {
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(threads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = chain ? 1 : 0;
  const cudaError_t e = cudaLaunchKernelEx(&cfg, kernel, static_cast<P>(args)...);
  if (e != cudaSuccess) {
    record_cuda_error(e);
    cudaGetLastError();
    return NASG_ERR_CUDA;
  }
  return NASG_OK;
}

template <int THREADS, int ITEMS, typename K, typename... A>
nasg_status launch_sort(K kernel, unsigned grid, cudaStream_t s, const A&... args) {
  constexpr size_t smem = sizeof(sort::Block<THREADS, ITEMS>);
  if (const nasg_status e = ensure_smem_limit(reinterpret_cast<const void*>(kernel), smem); e != NASG_OK) return e;
  return launch_chained(true, kernel, grid, THREADS, smem, s, args...);
}

template <int THREADS, int ITEMS>
nasg_status depth_sort(sort::Pass ps, Header* hdr, uint32_t* const dkeys[2], uint32_t* const order[2], uint32_t n,
                       cudaStream_t s) {
  const unsigned grid = unsigned(sort_blocks(n, kLargeDepth));
  const uint32_t* none = nullptr;
  for (int j = 0; j < kDepthPasses; ++j) {
    ps.hist = hdr->depth_hist[j];
    ps.ticket = hdr->tickets + j;
    ps.shift = 8 * j;
    ps.bits = 8;
    ps.tag = uint32_t(j + 1);
    const int i = j & 1;
    auto k = j == 0 ? depth_pass_kernel<THREADS, ITEMS, true, false>
                    : (j + 1 < kDepthPasses ? depth_pass_kernel<THREADS, ITEMS, false, false>
                                            : depth_pass_kernel<THREADS, ITEMS, false, true>);
    const nasg_status e = launch_sort<THREADS, ITEMS>(k, grid, s, ps, dkeys[i], j == 0 ? none : order[i], dkeys[1 - i],
                                                      order[1 - i], n, &hdr->drawn);
    if (e != NASG_OK) return e;
  }
  return NASG_OK;
}

// keys / vals[1] hold the result of an odd number of passes, [0] that of an even one.
template <int THREADS, int ITEMS>
nasg_status pair_sort(const ListArgs& la, sort::Pass ps, const TileDigits& td, int64_t most, uint32_t* const keys[2],
                      uint32_t* const vals[2], uint2* ranges, cudaStream_t s) {
  const unsigned grid = unsigned(sort_blocks(most, kLargePairs));
  for (int j = 0; j < td.passes; ++j) {
    ps.hist = la.hdr->tile_hist[j];
    ps.ticket = la.hdr->tickets + kDepthPasses + 1 + j;
    ps.shift = td.shift[j];
    ps.bits = td.bits[j];
    ps.tag = uint32_t(j + 1);
    const int i = j & 1;
    const bool last = j + 1 == td.passes;
    nasg_status e;
    if (j == 0) {
      auto k = last ? list_pass_kernel<THREADS, ITEMS, true> : list_pass_kernel<THREADS, ITEMS, false>;
      e = launch_sort<THREADS, ITEMS>(k, grid, s, la, ps, keys[1], vals[1], ranges);
    } else {
      auto k = last ? pair_pass_kernel<THREADS, ITEMS, true> : pair_pass_kernel<THREADS, ITEMS, false>;
      e = launch_sort<THREADS, ITEMS>(k, grid, s, la.hdr, ps, keys[i], vals[i], keys[1 - i], vals[1 - i], ranges,
                                      la.x_bits, la.tiles_x);
    }
    if (e != NASG_OK) return e;
  }
  return NASG_OK;
}

}  // namespace raster
}  // namespace nasg

using namespace nasg;
using namespace nasg::raster;

extern "C" size_t nasg_raster_workspace_bytes(int64_t n, int32_t width, int32_t height, int64_t max_pairs) {
  if (n < 0 || n >= (int64_t(1) << 31) || width < 1 || height < 1 || width > 16384 || height > 16384 ||
      max_pairs < 0 || max_pairs >= (int64_t(1) << 32))
    return 0;
  const int64_t tiles = int64_t((width + kTile - 1) / kTile) * ((height + kTile - 1) / kTile);
  return layout(n, tiles, int64_t(width) * height, max_pairs).total;
}

// `fail`: where the header's `failed` is set as by a wait that gave up (the probe's, else kNowhere).
enum FailAt { kNowhere, kBeforeSorts, kBeforeRender };

static nasg_status forward(FailAt fail, int64_t n, const float* means, const float* scales, const float* quats,
                           const float* opacity, const float* colours, const nasg_raster_camera* camera, float* image,
                           float* final_t, int64_t max_pairs, void* workspace, size_t workspace_bytes,
                           int64_t* n_pairs, void* stream) {
  if (!camera) return NASG_ERR_NULL;
  if (!camera_ok(camera)) return NASG_ERR_RANGE;
  if (n < 0 || n >= (int64_t(1) << 31) || max_pairs < 0 || max_pairs >= (int64_t(1) << 32)) return NASG_ERR_RANGE;
  if (!image || !final_t || !workspace) return NASG_ERR_NULL;
  if (n > 0 && (!means || !scales || !quats || !opacity || !colours)) return NASG_ERR_NULL;
  if (!aligned(workspace, 256) || !aligned(means, 4) || !aligned(image, 4) || !aligned(final_t, 4))
    return NASG_ERR_ALIGN;
  const Cam cam = make_cam(camera);
  const int64_t tiles = int64_t(cam.tx) * cam.ty;
  const int64_t pixels = int64_t(cam.w) * cam.h;
  const Layout L = layout(n, tiles, pixels, max_pairs);
  if (workspace_bytes < L.total) return NASG_ERR_RANGE;
  cudaStream_t s = as_stream(stream);
  unsigned char* ws = static_cast<unsigned char*>(workspace);
  auto at = [&](size_t off) { return reinterpret_cast<uint32_t*>(ws + off); };
  Header* hdr = reinterpret_cast<Header*>(ws + L.header);
  auto* splat = reinterpret_cast<Splat*>(ws + L.splat);
  auto* rows = reinterpret_cast<CoverRows*>(ws + L.rows);
  auto* rect = reinterpret_cast<uint2*>(ws + L.rect);
  uint32_t* reach = at(L.reach);
  auto* ranges = reinterpret_cast<uint2*>(ws + L.ranges);
  uint32_t* const keys[2] = {at(L.keys0), at(L.keys1)};
  uint32_t* const vals[2] = {at(L.vals0), at(L.vals1)};
  uint32_t* const dkeys[2] = {at(L.dkeys0), at(L.dkeys1)};
  uint32_t* const order[2] = {at(L.order0), at(L.order1)};
  const TileDigits td = tile_digits(cam.tx, cam.ty);

  if (cudaMemsetAsync(ws + L.header, 0, L.head_end - L.header, s) != cudaSuccess) return check_launch();
  auto* ncontrib = at(L.ncontrib);
  auto refuse = [&](nasg_status why) { return give_up(why, ncontrib, pixels, s); };
  auto set_failed = [&](FailAt where) {
    return fail != where || cudaMemsetAsync(&hdr->failed, 1, 1, s) == cudaSuccess;
  };
  if (!set_failed(kBeforeSorts)) return refuse(check_launch());
  unsigned long long total64 = 0;
  if (n > 0) {
    static thread_local HostWords host;
    if (!host.ready()) return refuse(check_launch());
    const unsigned long long call = ++host.calls;
    ProjectArgs pa{n, means, scales, quats, opacity, cam, td, splat, rows, rect, reach, dkeys[0], hdr, host.words, call};
    const int64_t blocks = (n + kBlock - 1) / kBlock;
    const int64_t most = int64_t(sm_count()) * 4;
    project_kernel<<<unsigned(blocks < most ? blocks : most), kBlock, 0, s>>>(pa);
    if (const nasg_status e = check_launch(); e != NASG_OK) return refuse(e);
    sort::Pass ps{};
    ps.states = reinterpret_cast<unsigned long long*>(ws + L.depth_states);
    ps.failed = &hdr->failed;
    ps.err = device_error_word();
    ps.limit = kWaitLimit;
    nasg_status e = n > kLargeDepth
                              ? depth_sort<kLargeThreads, kLargeItems>(ps, hdr, dkeys, order, uint32_t(n), s)
                              : depth_sort<kSmallThreads, kSmallItems>(ps, hdr, dkeys, order, uint32_t(n), s);
    if (e != NASG_OK) return refuse(e);
    constexpr int64_t kChunk = kBlock * kScanItems;
    e = launch_chained(true, offsets_kernel, unsigned((n + kChunk - 1) / kChunk), kBlock, 0, s, hdr,
                       hdr->tickets + kDepthPasses, ps.err, (unsigned long long)(max_pairs),
                       reinterpret_cast<ulonglong2*>(ws + L.pair_states),
                       reinterpret_cast<unsigned long long*>(ws + L.scan_states), order[kDepthPasses & 1], reach,
                       at(L.offsets), at(L.starts));
    if (e != NASG_OK) return refuse(e);
    // the host waits for the projection's total while the GPU sorts by depth
    if (!wait_total(host.words, call, s, &total64)) return refuse(NASG_ERR_CUDA);
  }
  if (n_pairs) *n_pairs = int64_t(total64);
  if (int64_t(total64) > max_pairs) return refuse(NASG_ERR_CAPACITY);
  if (total64 > 0) {
    const int64_t most = int64_t(total64);  // at least the pairs listed
    sort::Pass ps{};
    ps.states = reinterpret_cast<unsigned long long*>(ws + L.pair_states);
    ps.failed = &hdr->failed;
    ps.err = device_error_word();
    ps.limit = kWaitLimit;
    const ListArgs la{hdr, order[kDepthPasses & 1], at(L.offsets), at(L.starts), rect, reach, rows, td.x_bits, cam.tx};
    const nasg_status e = most > kLargePairs
                              ? pair_sort<kLargeThreads, kLargeItems>(la, ps, td, most, keys, vals, ranges, s)
                              : pair_sort<kSmallThreads, kSmallItems>(la, ps, td, most, keys, vals, ranges, s);
    if (e != NASG_OK) return refuse(e);
  }
  if (!set_failed(kBeforeRender)) return refuse(check_launch());
  const uint32_t* list = vals[td.passes & 1];
  const nasg_status e =
      two_pixels(tiles, 8)
          ? launch_chained(n > 0, render_fwd_kernel<2>, unsigned(tiles), TileShape<2>::NT, 0, s, cam, hdr, ranges, list,
                           splat, colours, image, final_t, ncontrib)
          : launch_chained(n > 0, render_fwd_kernel<1>, unsigned(tiles), TileShape<1>::NT, 0, s, cam, hdr, ranges, list,
                           splat, colours, image, final_t, ncontrib);
  return e == NASG_OK ? e : refuse(e);
}

extern "C" nasg_status nasg_raster_forward(int64_t n, const float* means, const float* scales, const float* quats,
                                           const float* opacity, const float* colours,
                                           const nasg_raster_camera* camera, float* image, float* final_t,
                                           int64_t max_pairs, void* workspace, size_t workspace_bytes,
                                           int64_t* n_pairs, void* stream) {
  return forward(kNowhere, n, means, scales, quats, opacity, colours, camera, image, final_t, max_pairs, workspace,
                 workspace_bytes, n_pairs, stream);
}

extern "C" nasg_status nasg_probe_raster_failed(int32_t where, int64_t n, const float* means, const float* scales,
                                                const float* quats, const float* opacity, const float* colours,
                                                const nasg_raster_camera* camera, float* image, float* final_t,
                                                int64_t max_pairs, void* workspace, size_t workspace_bytes,
                                                void* stream) {
  if (where != kBeforeSorts && where != kBeforeRender) return NASG_ERR_RANGE;
  return forward(FailAt(where), n, means, scales, quats, opacity, colours, camera, image, final_t, max_pairs, workspace,
                 workspace_bytes, nullptr, stream);
}

// ---------------------------------------------------------------------------
// Diagnostic: sort and scan blocks whose first predecessor never publishes
// ---------------------------------------------------------------------------
namespace nasg {
namespace raster {

constexpr int kProbeBlocks = NASG_PROBE_LOOK_BACK_BLOCKS;  // after block 0; more than a look-back reads at once

struct ProbeStates {
  unsigned long long sort[kProbeBlocks + 1][sort::kBins], scan[kProbeBlocks + 1];
};
static_assert(sizeof(ProbeStates) <= NASG_PROBE_LOOK_BACK_BYTES, "the header's size");

// results[b - 1]: entries that sort block b placed, or -1; results[kProbeBlocks + b - 1]: the scan's count
// before block b, or -1; results[2 kProbeBlocks]: the `failed` word.
__global__ void __launch_bounds__(kSmallThreads) look_back_probe_kernel(sort::Pass ps, int first,
                                                                       unsigned long long* scan, int32_t* results) {
  extern __shared__ __align__(16) unsigned char sort_smem[];
  auto& s = *reinterpret_cast<sort::Block<kSmallThreads, kSmallItems>*>(sort_smem);
  const uint32_t block = blockIdx.x + uint32_t(first);
  uint32_t key[kSmallItems], val[kSmallItems];
  for (int i = 0; i < kSmallItems; ++i) key[i] = val[i] = threadIdx.x + uint32_t(i) * kSmallThreads;
  const int placed = sort::sort_block<kSmallThreads, kSmallItems, false>(s, ps, block, 0u, key, val);
  if (threadIdx.x < 32) {
    if (threadIdx.x == 0) sort::st_state(scan + block, (block == 0 ? sort::kAll : sort::kOwn) | sort::tag_bits(ps.tag) | 1u);
    unsigned long long before = 0;
    const bool ok = block == 0 || sort::look_back_warp(scan, block, ps.tag, ps.limit, ps.err, &before);
    if (threadIdx.x == 0 && block > 0) {
      sort::st_state(scan + block, (ok ? sort::kAll : sort::kGone) | sort::tag_bits(ps.tag) | (before + 1u));
      results[block - 1] = placed;
      results[kProbeBlocks + block - 1] = ok ? int32_t(before) : -1;
    }
  }
}

}  // namespace raster
}  // namespace nasg

extern "C" nasg_status nasg_probe_look_back_timeout(int32_t limit, int32_t first, int32_t* results, void* workspace,
                                                    size_t workspace_bytes, void* stream) {
  if (limit < 1 || limit > (1 << 20) || (first != 0 && first != 1)) return NASG_ERR_RANGE;
  if (!results || !workspace) return NASG_ERR_NULL;
  if (!aligned(results, 4) || !aligned(workspace, 8)) return NASG_ERR_ALIGN;
  if (workspace_bytes < NASG_PROBE_LOOK_BACK_BYTES) return NASG_ERR_RANGE;
  cudaStream_t s = as_stream(stream);
  auto* states = static_cast<ProbeStates*>(workspace);
  if (cudaMemsetAsync(states, 0, sizeof(ProbeStates), s) != cudaSuccess ||
      cudaMemsetAsync(results, 0, (2 * kProbeBlocks + 1) * sizeof(int32_t), s) != cudaSuccess)
    return check_launch();
  sort::Pass ps{};
  ps.states = &states->sort[0][0];
  ps.failed = reinterpret_cast<uint32_t*>(results + 2 * kProbeBlocks);
  ps.err = device_error_word();
  ps.bits = 8;
  ps.tag = 1;
  ps.limit = uint32_t(limit);
  constexpr size_t smem = sizeof(sort::Block<kSmallThreads, kSmallItems>);
  if (const nasg_status e = ensure_smem_limit(reinterpret_cast<const void*>(look_back_probe_kernel), smem); e != NASG_OK)
    return e;
  look_back_probe_kernel<<<unsigned(kProbeBlocks + 1 - first), kSmallThreads, smem, s>>>(ps, first, states->scan, results);
  return check_launch();
}

extern "C" nasg_status nasg_raster_backward(int64_t n, const float* colours, const nasg_raster_camera* camera,
                                            const float* final_t, const float* g_image, float* g_colours,
                                            float* g_opacity, int64_t max_pairs, void* workspace,
                                            size_t workspace_bytes, void* stream) {
  if (!camera) return NASG_ERR_NULL;
  if (!camera_ok(camera)) return NASG_ERR_RANGE;
  if (n < 0 || n >= (int64_t(1) << 31) || max_pairs < 0 || max_pairs >= (int64_t(1) << 32)) return NASG_ERR_RANGE;
  if (!final_t || !g_image || !workspace || !g_colours || !g_opacity) return NASG_ERR_NULL;
  if (n > 0 && !colours) return NASG_ERR_NULL;
  if (!aligned(workspace, 256)) return NASG_ERR_ALIGN;
  const Cam cam = make_cam(camera);
  const int64_t tiles = int64_t(cam.tx) * cam.ty;
  const Layout L = layout(n, tiles, int64_t(cam.w) * cam.h, max_pairs);
  if (workspace_bytes < L.total) return NASG_ERR_RANGE;
  cudaStream_t s = as_stream(stream);
  unsigned char* ws = static_cast<unsigned char*>(workspace);
  if (cudaMemsetAsync(g_colours, 0, size_t(n) * 3 * sizeof(float), s) != cudaSuccess ||
      cudaMemsetAsync(g_opacity, 0, size_t(n) * sizeof(float), s) != cudaSuccess)
    return check_launch();
  if (n == 0) return NASG_OK;
  // the forward's sort ends in buffer (passes % 2)
  const uint32_t* vals = reinterpret_cast<const uint32_t*>(ws + (tile_digits(cam.tx, cam.ty).passes % 2 ? L.vals1 : L.vals0));
  const auto* hdr = reinterpret_cast<const Header*>(ws + L.header);
  const auto* ranges = reinterpret_cast<const uint2*>(ws + L.ranges);
  const auto* splat = reinterpret_cast<const Splat*>(ws + L.splat);
  const auto* ncontrib = reinterpret_cast<const uint32_t*>(ws + L.ncontrib);
  if (two_pixels(tiles, 4))
    render_bwd_kernel<2><<<unsigned(tiles), TileShape<2>::NT, 0, s>>>(cam, hdr, ranges, vals, splat, colours, final_t,
                                                                      ncontrib, g_image, g_colours, g_opacity);
  else
    render_bwd_kernel<1><<<unsigned(tiles), TileShape<1>::NT, 0, s>>>(cam, hdr, ranges, vals, splat, colours, final_t,
                                                                      ncontrib, g_image, g_colours, g_opacity);
  return check_launch();
}

// binning.cu -- tile-key duplication and sorting of (Gaussian, tile)
// instances, per frame of a batch.
//
// The instance order is that of a stable sort of the 64-bit keys
// (frame * tiles + tile) << 32 | bits(z), with instances emitted in Gaussian
// order (so equal keys stay in index order).  It is computed as an LSD radix
// sort whose low digits (the 32 depth bits) are applied to the Gaussians
// BEFORE duplication -- they are a per-Gaussian key -- and whose high digit
// (frame, tile) is one stable counting pass over the duplicated instances:
//   1. depth sort: 4 passes of 8 bits over the per-frame depth keys
//      (culled Gaussians carry 0xFFFFFFFF and are left out), each tile of
//      keys ranked in shared memory and written out in digit order; the last
//      pass also writes each Gaussian's tile rectangle in depth order;
//   2. tile masks: a warp takes 32 depth-consecutive Gaussians at a time (a
//      group); for each it sets the bits of the tile columns and rows that its
//      rectangle covers, and transposing these bits across the lanes gives, per
//      tile column and row, the 32-bit mask of the group's Gaussians on it.  The
//      Gaussians on a tile are the AND of its column's and its row's mask, in
//      depth order from the lowest bit;
//   3. per chunk (a run of groups of one frame), tile counts: the
//      masks' population counts summed over its groups; a scan over each frame's
//      chunks per tile, and over all tiles, gives the tile ranges;
//   4. scatter: the same masks again, each lane writing its tiles' Gaussians from
//      the tile's cursor on (stable by construction).
// The 64-bit keys themselves are never needed by the compositing kernels;
// gftorf_export_tile_lists materialises them from the ranges.
#include "gftorf_internal.cuh"

namespace gftorf {
namespace {

// Exclusive scan in place of a[0..S) by one CTA; returns the total through
// *total (if non-null).  Each thread scans a contiguous segment.
template <typename T>
__device__ void cta_exclusive_scan(T* a, int64_t S, uint64_t* total) {
  __shared__ uint64_t s_warp[32];
  const int nt = blockDim.x, tid = threadIdx.x;
  const int64_t seg = (S + nt - 1) / nt;
  const int64_t lo = min((int64_t)tid * seg, S), hi = min(lo + seg, S);
  uint64_t sum = 0;
  for (int64_t i = lo; i < hi; ++i) sum += a[i];
  // block exclusive scan of the segment sums
  const int lane = tid & 31, wid = tid >> 5;
  uint64_t incl = sum;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    uint64_t v = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += v;
  }
  if (lane == 31) s_warp[wid] = incl;
  __syncthreads();
  if (wid == 0) {
    const int nw = (nt + 31) / 32;
    uint64_t v = lane < nw ? s_warp[lane] : 0;
    uint64_t x = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      uint64_t y = __shfl_up_sync(0xffffffffu, x, o);
      if (lane >= o) x += y;
    }
    if (lane < nw) s_warp[lane] = x - v;  // exclusive warp offsets
  }
  __syncthreads();
  uint64_t run = s_warp[wid] + incl - sum;
  for (int64_t i = lo; i < hi; ++i) {
    const uint64_t v = a[i];
    a[i] = (T)run;
    run += v;
  }
  if (total && tid == nt - 1) *total = run;
  __syncthreads();
}

// ---------------------------------------------------------------------------
// tile masks of a group of 32 Gaussians
// ---------------------------------------------------------------------------
__device__ __forceinline__ uint32_t shl_clamp(uint32_t x, int n) {  // 0 for n >= 32
  uint32_t r;
  asm("shl.b32 %0, %1, %2;" : "=r"(r) : "r"(x), "r"(n));
  return r;
}
// bits [lo, hi) of an endless bit string, word w
__device__ __forceinline__ uint32_t span_word(int lo, int hi, int w) {
  const uint32_t from = shl_clamp(0xFFFFFFFFu, max(lo - 32 * w, 0));
  return from & ~shl_clamp(0xFFFFFFFFu, max(hi - 32 * w, 0));
}
// lane l's bit g <- lane g's bit l
__device__ __forceinline__ uint32_t transpose32(uint32_t x, int lane) {
  uint32_t m = 0x0000FFFFu;  // the bits whose index has bit j clear
#pragma unroll
  for (int j = 16; j > 0; j >>= 1) {
    const uint32_t y = __shfl_xor_sync(0xffffffffu, x, j);
    x = lane & j ? (x & ~m) | ((y >> j) & m) : (x & m) | ((y & m) << j);
    m ^= m << (j >> 1);
  }
  return x;
}
// words of a warp's masks: one per tile column, then one per tile row, padded
__host__ __device__ constexpr int mask_words(int tiles_x, int tiles_y) {
  return (tiles_x + tiles_y + 31) / 32 * 32;
}
// the masks of the group whose lane-th Gaussian covers the rectangle rr, by a warp
__device__ __forceinline__ void group_masks(uint32_t* masks, uint2 rr, int tiles_x, int words,
                                            int lane) {
  int x0, y0, x1, y1;
  unpack_rect(rr, x0, y0, x1, y1);
  for (int w = 0; w < words; w += 32)
    masks[w + lane] = transpose32(span_word(x0, x1, w >> 5) |
                                      span_word(tiles_x + y0, tiles_x + y1, w >> 5), lane);
}

// ---------------------------------------------------------------------------
// footprints given by the caller (binning-only entry point)
// ---------------------------------------------------------------------------
__global__ void footprint_kernel(const float* __restrict__ u,
                                 const float* __restrict__ v,
                                 const int32_t* __restrict__ radius,
                                 const float* __restrict__ z,
                                 Header* __restrict__ hdr,
                                 uint2* __restrict__ rect,
                                 uint32_t* __restrict__ zkey, int N, int TW,
                                 int TH, int tiles_x, int tiles_y) {
  grid_begin_early();
  const int g = blockIdx.x * blockDim.x + threadIdx.x;
  const int b = blockIdx.y;
  bool visible = false;
  if (g < N) {
    const size_t i = (size_t)b * N + g;
    uint2 rr = make_uint2(0, 0);
    uint32_t key = kCulledKey;
    const int r = radius[i];
    if (r > 0) {
      int x0, y0, x1, y1;
      tile_rect(u[i], v[i], r, TW, TH, tiles_x, tiles_y, x0, y0, x1, y1);
      if (x0 < x1 && y0 < y1) {
        visible = true;
        rr = pack_rect(x0, y0, x1, y1);
        key = __float_as_uint(z[i]);
      }
    }
    rect[i] = rr;
    zkey[i] = key;
  }
  const unsigned m = __ballot_sync(0xffffffffu, visible);
  if ((threadIdx.x & 31) == 0 && m) atomicAdd(&hdr->vis[b], (uint32_t)__popc(m));
}

// Most tiles that discs of the given radii can meet, summed
__global__ void __launch_bounds__(256)
    footprint_bound_kernel(const int32_t* __restrict__ radius, int64_t n, int TW, int TH,
                           unsigned long long* __restrict__ bound) {
  grid_begin_early();
  __shared__ unsigned long long s_sum[8];
  unsigned long long sum = 0;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x) {
    const uint32_t d = 2u * (uint32_t)max(radius[i], 0);  // below 2^32
    sum += (unsigned long long)(d / (uint32_t)TW + 2u) * (d / (uint32_t)TH + 2u);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
  if ((threadIdx.x & 31) == 0) s_sum[threadIdx.x >> 5] = sum;
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 1; w < 8; ++w) sum += s_sum[w];
    if (sum) atomicAdd(bound, sum);
  }
}

// ---------------------------------------------------------------------------
// depth sort: stable LSD radix sort, 8-bit digits, one segment per frame.
// The per-frame digit totals of all four passes come from one reading of the
// keys (they do not depend on the order); each pass is then one kernel that
// ranks a tile of keys in shared memory and finds the tile's offset for each
// digit from the tiles before it (decoupled look-back: every tile publishes
// its digit counts, then the running prefix once it knows it).  Culled
// Gaussians (key 0xFFFFFFFF) are left out: their place in the order is never
// read (every later kernel stops at the frame's visible count), so the first
// pass packs the visible keys at the front of the frame and the later passes
// run only the frame's ceil(visible / 2048) tiles.
// ---------------------------------------------------------------------------
constexpr uint32_t kLbPrefix = 0x80000000u;  // status word: inclusive prefix
constexpr uint32_t kLbAggregate = 0x40000000u;  // status word: this tile's count only
constexpr uint32_t kLbCount = 0x3FFFFFFFu;
constexpr int kLbSpinLimit = 1 << 22;  // bounded wait on a predecessor tile

__global__ void __launch_bounds__(kSortThreads)
    dsort_hist_kernel(const uint32_t* __restrict__ keys, int N, uint32_t* __restrict__ ghist) {
  grid_begin_early();
  __shared__ uint32_t h[4][256];
  const int blk = blockIdx.x, b = blockIdx.y, tid = threadIdx.x;
  for (int i = tid; i < 4 * 256; i += kSortThreads) (&h[0][0])[i] = 0;
  __syncthreads();
  const uint32_t* k = keys + (size_t)b * N;
#pragma unroll
  for (int it = 0; it < kSortItems; ++it) {
    const int pos = blk * kSortTile + it * kSortThreads + tid;
    if (pos < N) {
      const uint32_t key = k[pos];
      if (key != kCulledKey) {
#pragma unroll
        for (int p = 0; p < 4; ++p) atomicAdd(&h[p][(key >> (8 * p)) & 255u], 1u);
      }
    }
  }
  __syncthreads();
  for (int i = tid; i < 4 * 256; i += kSortThreads) {
    const uint32_t c = (&h[0][0])[i];
    if (c) atomicAdd(&ghist[(size_t)b * 1024 + i], c);
  }
}

// per (frame, pass): exclusive scan of the 256 digit totals -> digit bases
__global__ void __launch_bounds__(256) dsort_bases_kernel(uint32_t* __restrict__ ghist) {
  grid_begin_early();
  cta_exclusive_scan<uint32_t>(ghist + (size_t)blockIdx.x * 256, 256, nullptr);
}

// One pass: tiles are claimed in order through an atomic counter, so a tile
// only ever waits for tiles that are already running.  rin/rout (last pass
// only, else null): the Gaussians' tile rectangles are written in the
// sorted order as well.
__global__ void __launch_bounds__(kSortThreads, 5)  // <= 48 registers, no spill
    dsort_pass_kernel(const uint32_t* __restrict__ kin, const uint32_t* __restrict__ iin,
                      uint32_t* __restrict__ kout, uint32_t* __restrict__ iout, int N, int B,
                      int pass, int n_dblk, const uint32_t* __restrict__ gbase,
                      uint32_t* __restrict__ status, uint32_t* __restrict__ tile_counter,
                      Header* __restrict__ hdr, const uint2* __restrict__ rin,
                      uint2* __restrict__ rout) {
  grid_begin_early();
  __shared__ uint32_t wc[kSortWarps][256];
  __shared__ uint32_t s_tile;
  // the tile's keys and indices in digit order (staged, then written out in
  // runs of consecutive places), each digit's first place in the tile and in
  // the frame, the warps' digit-count sums
  __shared__ uint32_t s_key[kSortTile], s_id[kSortTile];
  __shared__ uint32_t s_tstart[256], s_gbase[256], s_wsum[kSortWarps];
  const int tid = threadIdx.x, w = tid >> 5, lane = tid & 31;
  const int shift = 8 * pass;
  if (tid == 0) s_tile = atomicAdd(tile_counter, 1u);
  for (int i = tid; i < kSortWarps * 256; i += kSortThreads) (&wc[0][0])[i] = 0;
  __syncthreads();
  const uint32_t L = s_tile;
  const int b = (int)(L / (uint32_t)n_dblk), blk = (int)(L - (uint32_t)b * n_dblk);
  const size_t fb = (size_t)b * N;
  const int start = blk * kSortTile + w * (kSortTile / kSortWarps);
  // the first pass reads all N keys of the frame (culled ones skipped), the
  // later ones the visible keys packed at its front
  const int vis = (int)hdr->vis[b];
  const int n_in = pass == 0 ? N : vis;
  if (blk * kSortTile >= n_in) return;  // no keys: no later tile waits for it
  uint32_t key[kSortItems], id[kSortItems], loc[kSortItems];
  bool live[kSortItems];
#pragma unroll
  for (int it = 0; it < kSortItems; ++it) {  // all loads in flight first
    const int pos = start + it * 32 + lane;
    const bool valid = pos < n_in;
    key[it] = valid ? kin[fb + pos] : kCulledKey;
    id[it] = valid ? (iin ? iin[fb + pos] : (uint32_t)pos) : 0u;
  }
#pragma unroll
  for (int it = 0; it < kSortItems; ++it) live[it] = key[it] != kCulledKey;
  // rank within the warp (lanes in order, items in order): stable.  The
  // lanes sharing a digit in each item first (independent of one another:
  // eight ballots, one per digit bit, measured faster than match.any), then
  // the warp's running digit counts item after item.
  uint32_t peers[kSortItems];
  const uint32_t lt = lanemask_lt();
#pragma unroll
  for (int it = 0; it < kSortItems; ++it) {
    // lanes with the same digit: one ballot per digit bit (live lanes only)
    const uint32_t d = (key[it] >> shift) & 255u;
    unsigned pm = __ballot_sync(0xffffffffu, live[it]);
#pragma unroll
    for (int bit = 0; bit < 8; ++bit) {
      const bool on = (d >> bit) & 1u;
      const unsigned bm = __ballot_sync(0xffffffffu, on);
      pm &= on ? bm : ~bm;
    }
    peers[it] = live[it] ? pm : (1u << lane);
  }
#pragma unroll
  for (int it = 0; it < kSortItems; ++it) {
    const bool valid = live[it];
    const uint32_t d = (key[it] >> shift) & 255u;
    const uint32_t rank = __popc(peers[it] & lt);
    const uint32_t before = valid ? wc[w][d] : 0u;
    __syncwarp();
    if (valid && rank == 0) wc[w][d] = before + __popc(peers[it]);
    __syncwarp();
    loc[it] = before + rank;
  }
  __syncthreads();
  {
    const int d = tid;  // 256 threads, one digit each
    uint32_t cnt = 0;
#pragma unroll
    for (int ww = 0; ww < kSortWarps; ++ww) {
      const uint32_t t = wc[ww][d];
      wc[ww][d] = cnt;
      cnt += t;
    }
    // publish this tile's count, then find the count of the tiles before it
    volatile uint32_t* st = status + ((size_t)pass * B + b) * (size_t)n_dblk * 256;
    uint32_t excl = 0;
    if (blk == 0) {
      st[d] = kLbPrefix | cnt;
    } else {
      st[(size_t)blk * 256 + d] = kLbAggregate | cnt;
      int j = blk - 1, spins = 0;
      for (;;) {
        const uint32_t v = st[(size_t)j * 256 + d];
        if (v == 0u) {
          if (++spins > kLbSpinLimit) {  // never expected: tiles before are running
            set_status(hdr, GFTORF_ERR_TIMEOUT);
            break;
          }
          __nanosleep(32);
          continue;
        }
        excl += v & kLbCount;
        if ((v & kLbPrefix) || j == 0) break;
        --j;
      }
      st[(size_t)blk * 256 + d] = kLbPrefix | (excl + cnt);
    }
    s_gbase[d] = gbase[((size_t)b * 4 + pass) * 256 + d] + excl;
    // first place of digit d in the tile: exclusive scan of the counts
    uint32_t incl = cnt;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t y = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl += y;
    }
    if (lane == 31) s_wsum[w] = incl;
    __syncthreads();
    uint32_t before = 0;
#pragma unroll
    for (int ww = 0; ww < kSortWarps; ++ww) before += ww < w ? s_wsum[ww] : 0u;
    s_tstart[d] = before + incl - cnt;
  }
  __syncthreads();
  // stage in digit order: place = digit start + earlier warps' count of the
  // digit + rank in the warp
#pragma unroll
  for (int it = 0; it < kSortItems; ++it) {
    if (live[it]) {
      const uint32_t d = (key[it] >> shift) & 255u;
      const uint32_t tp = s_tstart[d] + wc[w][d] + loc[it];
      s_key[tp] = key[it];
      s_id[tp] = id[it];
    }
  }
  __syncthreads();
  // write out: consecutive threads take consecutive staged places, which lie
  // in runs of one digit at consecutive places of the frame
  uint32_t n_live = 0;
#pragma unroll
  for (int ww = 0; ww < kSortWarps; ++ww) n_live += s_wsum[ww];
  if (!rout) {
    for (uint32_t p = tid; p < n_live; p += kSortThreads) {
      const uint32_t k = s_key[p], g = s_id[p];
      const uint32_t d = (k >> shift) & 255u;
      const uint32_t dst = s_gbase[d] + (p - s_tstart[d]);
      if (dst < (uint32_t)vis) {  // always (a timed-out wait leaves garbage, not a fault)
        kout[fb + dst] = k;
        iout[fb + dst] = g;
      }
    }
    return;
  }
  // last pass: indices and rectangles in depth order (the keys
  // are not needed again); the rectangles' gathers of four places at once
  constexpr int G = 4;
#pragma unroll 1
  for (uint32_t p0 = tid; p0 < n_live; p0 += G * kSortThreads) {
    uint32_t gg[G], dd[G];
    uint2 rr[G];
#pragma unroll
    for (int i = 0; i < G; ++i) {
      const uint32_t p = p0 + i * kSortThreads;
      dd[i] = 0xFFFFFFFFu;
      gg[i] = 0u;
      rr[i] = make_uint2(0u, 0u);
      if (p < n_live) {
        const uint32_t k = s_key[p], g = s_id[p];
        const uint32_t d = (k >> shift) & 255u;
        const uint32_t dst = s_gbase[d] + (p - s_tstart[d]);
        // always (a timed-out wait leaves garbage, not a fault)
        if (dst < (uint32_t)vis && g < (uint32_t)N) {
          dd[i] = dst;
          gg[i] = g;
          rr[i] = rin[fb + g];
        }
      }
    }
#pragma unroll
    for (int i = 0; i < G; ++i) {
      if (dd[i] != 0xFFFFFFFFu) {
        iout[fb + dd[i]] = gg[i];
        rout[fb + dd[i]] = rr[i];
      }
    }
  }
}

// ---------------------------------------------------------------------------
// chunk counts, column scan and scatter.  A chunk is L.chunk depth-consecutive
// Gaussians of a frame (a multiple of 32); chunk c of frame b has row b n_chunk + c
// of the counts.
//
// Small grids (below kBlockTiles tiles): a CTA takes L.chunks_per_cta chunks: its warps
// form the masks of their groups over the whole grid, then every thread takes (chunk,
// tile) items, walking the chunk's groups with the count or the cursor in a register.
// (Chunks of instances, from a scan of the Gaussians' tile counts, with one
// instance per lane and the lanes of one tile ranked by match.any, executed 4.4
// instructions per instance on a chain of shared-memory cursor updates: scan,
// count, column scan and scatter 144 us for 16 frames of 300k Gaussians at 64x64
// tiles, now 109; one frame of 100k at 32x32 51 and now 29.  One warp per chunk with
// its cursors in shared memory instead of items: 116, 46.)
//
// Larger grids: a CTA takes one chunk and one block of tiles, of at most 32 columns and
// rows together (64 on grids of kWideBlocks such blocks and more), first packs those of
// its Gaussians that meet the block, in order, and forms the masks of these alone, one
// word (two) per lane and group of 32.  Over the whole grid the work grows with
// Gaussians x tiles, whatever the footprints, and few CTAs do it where the space for
// the counts allows few chunks: 300k Gaussians of radius 1 to 3 on 3840x2160 at 16x16
// tiles, the whole binning 8255 us, in blocks 142; 12 frames of 120k on 517x389 at
// 16x16 (lists of 40 tiles per Gaussian) 227 and 195; 16 of 300k at 32x32 (300 tiles)
// 348 and 321.  At 180 tiles (64x32) a word holds nearly the grid.
// ---------------------------------------------------------------------------
struct ChunkArgs {
  int N, NT, tiles_x, tiles_y, chunk, n_chunk, per_cta;
  int bw, bh, blocks_x, n_block;  // of the blocks of tiles (0: the whole grid)
};

// masks (and indices, if ids) of the CTA's groups, group g the Gaussians r0 + 32 g ..
// + 31 of the frame's depth order, empty from r1 on
__device__ __forceinline__ void grid_masks(uint32_t* smem, int stride, const uint2* rc,
                                           const uint32_t* id, int r0, int r1, int groups,
                                           int tiles_x, int words) {
  const int lane = threadIdx.x & 31, nw = blockDim.x >> 5;
  for (int g = threadIdx.x >> 5; g < groups; g += nw) {
    const int r = r0 + 32 * g + lane;
    uint32_t* m = smem + (size_t)g * stride;
    const uint2 rr = r < r1 ? rc[r] : make_uint2(0u, 0u);
    if (id) m[words + lane] = r < r1 ? id[r] : 0u;
    group_masks(m, rr, tiles_x, words, lane);
  }
  __syncthreads();
}

constexpr int kBinThreads = 256;

__global__ void __launch_bounds__(kBinThreads)
    tile_count_kernel(const uint2* __restrict__ srect, const Header* __restrict__ hdr,
                      uint32_t* __restrict__ tcnt, ChunkArgs a) {
  grid_begin_early();
  extern __shared__ uint32_t smem[];
  const int b = blockIdx.y, c0 = blockIdx.x * a.per_cta, vis = (int)hdr->vis[b];
  const int r0 = c0 * a.chunk, r1 = min(r0 + a.per_cta * a.chunk, vis);
  if (r0 >= r1) return;
  const int words = mask_words(a.tiles_x, a.tiles_y), per = a.chunk / 32;
  const int groups = (r1 - r0 + 31) / 32, chunks = (r1 - r0 + a.chunk - 1) / a.chunk;
  grid_masks(smem, words, srect + (size_t)b * a.N, nullptr, r0, r1, groups, a.tiles_x, words);
  uint32_t* rows = tcnt + ((size_t)b * a.n_chunk + c0) * a.NT;
  for (int i = threadIdx.x; i < chunks * a.NT; i += kBinThreads) {
    const int c = i / a.NT, t = i - c * a.NT;
    const int ty = t / a.tiles_x, tx = t - ty * a.tiles_x;
    const int n = min(per, groups - c * per);
    const uint32_t *col = smem + c * per * words + tx, *row = col - tx + a.tiles_x + ty;
    uint32_t acc = 0;
#pragma unroll 8
    for (int g = 0; g < n; ++g, col += words, row += words) acc += __popc(*col & *row);
    rows[i] = acc;
  }
}

// A block of tiles [x, x + w) x [y, y + h)
struct TileBlock {
  int x, y, w, h;
};
__device__ __forceinline__ TileBlock tile_block(int k, const ChunkArgs& a) {
  TileBlock t;
  const int by = k / a.blocks_x;
  t.x = (k - by * a.blocks_x) * a.bw;
  t.y = by * a.bh;
  t.w = min(a.bw, a.tiles_x - t.x);
  t.h = min(a.bh, a.tiles_y - t.y);
  return t;
}
// The tiles a thread takes of a block with W words of columns and rows (at most
// 256 W^2 tiles): every 256th, as (column, row) in the block, and its index in the grid
template <int W>
struct OwnTiles {
  int tx[W * W], ty[W * W], tile[W * W];
  int n;
  __device__ __forceinline__ OwnTiles(const TileBlock& t, int tiles_x) {
    n = 0;
#pragma unroll
    for (int k = 0; k < W * W; ++k) {
      const int i = (int)threadIdx.x + k * kBinThreads;
      ty[k] = i / t.w;
      tx[k] = i - ty[k] * t.w;
      tile[k] = (t.y + ty[k]) * tiles_x + t.x + tx[k];
      n += ty[k] < t.h ? 1 : 0;
    }
  }
};

// The masks of those of the Gaussians [base, min(base + kBlockBatch, r1)) that meet the
// block, packed in order: word S g + l is column l of group g, or row l - w (W words of
// 32), and word S g + 64 + l the index of its l-th Gaussian (S = 96 words, with indices,
// or 64).
// Returns the number of groups; the whole CTA calls it, and may read the words until it
// calls again.  `in` holds the batch's rectangles and indices and gets the next one's,
// loaded while this one is worked on.
constexpr int kBlockBatch = 4 * kBinThreads;
template <int S>
struct BlockBatch {
  uint2 rect[4];  // four groups of 32 consecutive Gaussians per warp
  uint32_t id[4];
  __device__ __forceinline__ void load(const uint2* __restrict__ rc,
                                       const uint32_t* __restrict__ ids, int base, int r1) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int r = base + warp * 128 + 32 * i + lane;
      rect[i] = r < r1 ? rc[r] : make_uint2(0u, 0u);
      if (S == 96) id[i] = r < r1 ? ids[r] : 0u;
    }
  }
};
template <int W, int S>
__device__ __forceinline__ int block_masks(uint32_t* s_group, int* s_cnt, BlockBatch<S>& in,
                                           const uint2* __restrict__ rc,
                                           const uint32_t* __restrict__ ids, int base, int r1,
                                           const TileBlock& t) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  // both coordinates of a corner at once, tiles being fewer than 2^15: the top bit of
  // each half stays where first <= last tile of the block, or end > its first
  constexpr uint32_t kTop = 0x80008000u;
  const uint32_t last = (uint32_t)((t.x + t.w - 1) | (t.y + t.h - 1) << 16) | kTop;
  const uint32_t next = (uint32_t)((t.x + 1) | (t.y + 1) << 16);
  unsigned kept[4];
  int n = 0;
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const uint2 rr = in.rect[i];
    const bool meets = ((last - rr.x) & ((rr.y | kTop) - next) & kTop) == kTop;
    kept[i] = __ballot_sync(0xffffffffu, meets);
    n += __popc(kept[i]);
  }
  if (lane == 0) s_cnt[warp] = n;
  __syncthreads();  // (the previous batch's words have been read, too)
  int pos = 0, total = 0;
#pragma unroll
  for (int w = 0; w < kBinThreads / 32; ++w) {
    const int c = s_cnt[w];
    pos += w < warp ? c : 0;
    total += c;
  }
  if (n > 0) {
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      if (kept[i] >> lane & 1u) {
        const int at = pos + __popc(kept[i] & ((1u << lane) - 1u));
        uint32_t* d = s_group + (at >> 5) * S + (at & 31);
        d[0] = in.rect[i].x;
        d[32] = in.rect[i].y;
        if (S == 96) d[64] = in.id[i];
      }
      pos += __popc(kept[i]);
    }
  }
  in.load(rc, ids, base + kBlockBatch, r1);
  __syncthreads();
  const int groups = (total + 31) / 32;
  for (int g = warp; g < groups; g += kBinThreads / 32) {
    uint32_t* d = s_group + g * S + lane;
    int x0, y0, x1, y1;
    unpack_rect(32 * g + lane < total ? make_uint2(d[0], d[32]) : make_uint2(0u, 0u), x0, y0, x1,
                y1);
    x0 = max(x0 - t.x, 0), x1 = min(x1 - t.x, t.w);
    y0 = t.w + max(y0 - t.y, 0), y1 = t.w + min(y1 - t.y, t.h);
    if (32 * g + lane >= total) x1 = x0 = 0, y1 = y0 = 0;
#pragma unroll
    for (int k = 0; k < W; ++k)
      d[32 * k] = transpose32(span_word(x0, x1, k) | span_word(y0, y1, k), lane);
  }
  __syncthreads();
  return groups;
}

template <int W>
__global__ void __launch_bounds__(kBinThreads)
    block_count_kernel(const uint2* __restrict__ srect, const Header* __restrict__ hdr,
                       uint32_t* __restrict__ tcnt, uint64_t* __restrict__ sums, int n_sums,
                       ChunkArgs a) {
  grid_begin_early();
  if (blockIdx.x == 0 && blockIdx.y == 0)  // for the column scan
    for (int i = threadIdx.x; i < n_sums; i += kBinThreads) sums[i] = 0u;
  __shared__ uint32_t s_group[kBlockBatch * 2];
  __shared__ int s_cnt[kBinThreads / 32];
  const int b = blockIdx.y, c = blockIdx.x / a.n_block, vis = (int)hdr->vis[b];
  const int r0 = c * a.chunk, r1 = min(r0 + a.chunk, vis);
  if (r0 >= r1) return;
  const TileBlock t = tile_block(blockIdx.x - c * a.n_block, a);
  const OwnTiles<W> own(t, a.tiles_x);
  const uint2* rc = srect + (size_t)b * a.N;
  uint32_t acc[W * W];
#pragma unroll
  for (int k = 0; k < W * W; ++k) acc[k] = 0;
  BlockBatch<64> in;
  in.load(rc, nullptr, r0, r1);
  for (int base = r0; base < r1; base += kBlockBatch) {
    const int groups = block_masks<W, 64>(s_group, s_cnt, in, rc, nullptr, base, r1, t);
#pragma unroll
    for (int k = 0; k < W * W; ++k) {
      if (k >= own.n) break;
      const uint32_t *col = s_group + own.tx[k], *row = s_group + t.w + own.ty[k];
#pragma unroll 4
      for (int g = 0; g < groups; ++g) acc[k] += __popc(col[64 * g] & row[64 * g]);
    }
  }
  uint32_t* rows = tcnt + ((size_t)b * a.n_chunk + c) * a.NT;
#pragma unroll
  for (int k = 0; k < W * W; ++k)
    if (k < own.n) rows[own.tile[k]] = acc[k];
}

// Exclusive scan over the CTA of four consecutive totals per thread, added to base;
// base becomes the total's end, the same in every thread.
constexpr int kColWarps = 32, kColWarpsMany = 8;
constexpr int kScanTotals = 4 * 32 * kColWarps;  // per step
__device__ __forceinline__ uint64_t scan_totals(const uint32_t* __restrict__ ttot, int i, int n,
                                                uint32_t* v, uint64_t* s_w, uint64_t& base) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
#pragma unroll
  for (int k = 0; k < 4; ++k) v[k] = i + k < n ? __ldcg(&ttot[i + k]) : 0u;
  const uint64_t mine = (uint64_t)v[0] + v[1] + v[2] + v[3];
  uint64_t incl = mine;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint64_t y = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += y;
  }
  __syncthreads();  // s_w has been read
  if (lane == 31) s_w[w] = incl;
  __syncthreads();
  uint64_t st = base + incl - mine;
  for (int k = 0; k < kColWarps; ++k) {
    const uint64_t x = s_w[k];
    base += x;
    st += k < w ? x : 0u;
  }
  return st;
}
// the ranges of four consecutive tiles from the first one's start
__device__ __forceinline__ void put_ranges(uint2* __restrict__ ranges, int i, int n, uint64_t st,
                                           const uint32_t* v) {
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    if (i + k < n) ranges[i + k] = make_uint2((uint32_t)st, (uint32_t)(st + v[k]));
    st += v[k];
  }
}

// per (frame, tile): exclusive prefix over the frame's chunks, and the tile's total.
// A CTA covers 32 tiles (lanes, coalesced rows) and splits the frame's chunks into
// WARPS consecutive segments (warps): segment sums, then per-segment rescan.
// The CTA that finishes last makes the instance count, and with few tiles (kColWarps)
// scans the totals of all (frame, tile) in order, which gives the ranges; lists that
// overflow the capacity are left empty.  With many (kColWarpsMany) it scans only the sums of runs of
// kScanTotals tiles, which the CTAs have added up, and tile_range_kernel makes the
// ranges (16 frames of 8160 tiles, the binning: 514 -> 422 us; at five steps of
// kScanTotals 207 -> 192).
template <int WARPS>
__global__ void __launch_bounds__(32 * WARPS)
    tile_colscan_kernel(uint32_t* __restrict__ tcnt, uint32_t* __restrict__ ttot,
                        uint2* __restrict__ ranges, uint64_t* __restrict__ sums,
                        Header* __restrict__ hdr, ChunkArgs a, int64_t cap) {
  grid_begin_early();
  __shared__ uint32_t s_seg[WARPS][32];
  __shared__ uint64_t s_w[WARPS];
  __shared__ bool s_last;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int t = blockIdx.x * 32 + lane, b = blockIdx.y;
  const uint32_t n = ((uint32_t)hdr->vis[b] + a.chunk - 1) / a.chunk;
  const uint32_t seg = (n + WARPS - 1) / WARPS;
  const uint32_t s0 = min(n, (uint32_t)w * seg), s1 = min(n, (uint32_t)(w + 1) * seg);
  uint32_t* col = tcnt + (size_t)b * a.n_chunk * a.NT + t;
  uint32_t sum = 0;
  if (t < a.NT) {
#pragma unroll 8
    for (uint32_t c = s0; c < s1; ++c) sum += col[(size_t)c * a.NT];
  }
  s_seg[w][lane] = sum;
  __syncthreads();
  uint32_t run = 0;
  for (int ww = 0; ww < w; ++ww) run += s_seg[ww][lane];
  if (t < a.NT) {
#pragma unroll 8
    for (uint32_t c = s0; c < s1; ++c) {
      const uint32_t v = col[(size_t)c * a.NT];
      col[(size_t)c * a.NT] = run;
      run += v;
    }
    if (w == WARPS - 1) ttot[(size_t)b * a.NT + t] = run;
  }
  if (w == WARPS - 1) {
    if constexpr (WARPS == kColWarpsMany) {  // (32 consecutive tiles lie in one run or in two)
      const int i = b * a.NT + t, k = i / kScanTotals, k0 = __shfl_sync(0xffffffffu, k, 0);
      uint64_t lo = t < a.NT && k == k0 ? run : 0u, hi = t < a.NT && k != k0 ? run : 0u;
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        lo += __shfl_xor_sync(0xffffffffu, lo, o);
        hi += __shfl_xor_sync(0xffffffffu, hi, o);
      }
      if (lane == 0) {
        if (lo) atomicAdd(reinterpret_cast<unsigned long long*>(&sums[k0]), lo);
        if (hi) atomicAdd(reinterpret_cast<unsigned long long*>(&sums[k0 + 1]), hi);
      }
    }
    __threadfence();  // the totals' writers (the rest is for later kernels)
  }
  __syncthreads();
  if (threadIdx.x == 0)
    s_last = atomicAdd(&hdr->col_done, 1u) == gridDim.x * gridDim.y - 1;
  __syncthreads();
  if (!s_last) return;
  __threadfence();
  const int total_tiles = gridDim.y * a.NT;
  uint64_t base = 0;
  if constexpr (WARPS == kColWarpsMany) {  // at most 800 runs: four per thread
    const int runs = (total_tiles + kScanTotals - 1) / kScanTotals, i = 4 * (int)threadIdx.x;
    uint64_t v[4], mine = 0;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      v[k] = i + k < runs ? __ldcg(&sums[i + k]) : 0u;
      mine += v[k];
    }
    uint64_t incl = mine;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint64_t y = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl += y;
    }
    if (lane == 31) s_w[w] = incl;
    __syncthreads();
    uint64_t st = incl - mine;
    for (int k = 0; k < WARPS; ++k) {
      const uint64_t x = s_w[k];
      base += x;
      st += k < w ? x : 0u;
    }
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      if (i + k < runs) sums[i + k] = st;
      st += v[k];
    }
  } else {
    for (int i0 = 0; i0 < total_tiles; i0 += kScanTotals) {
      uint32_t v[4];
      const int i = i0 + 4 * threadIdx.x;
      const uint64_t st = scan_totals(ttot, i, total_tiles, v, s_w, base);
      put_ranges(ranges, i, total_tiles, st, v);
    }
  }
  const bool over = base > (uint64_t)cap;  // (the same base in every thread)
  if (over && WARPS == kColWarps)
    for (int i0 = 0; i0 < total_tiles; i0 += kScanTotals)  // a thread's own ranges
      for (int k = 0; k < 4; ++k)
        if (i0 + 4 * (int)threadIdx.x + k < total_tiles)
          ranges[i0 + 4 * threadIdx.x + k] = make_uint2(0u, 0u);
  if (threadIdx.x == 0) {
    hdr->count = (int64_t)base;
    if (over) set_status(hdr, GFTORF_ERR_CAPACITY);
    hdr->col_done = 0;  // for the next binning
  }
}

// the ranges of a run of kScanTotals tiles per CTA, from the run's start
__global__ void __launch_bounds__(32 * kColWarps)
    tile_range_kernel(const uint32_t* __restrict__ ttot, const uint64_t* __restrict__ sums,
                      const Header* __restrict__ hdr, uint2* __restrict__ ranges, int total_tiles,
                      int64_t cap) {
  grid_begin_early();
  __shared__ uint64_t s_w[kColWarps];
  const int i = blockIdx.x * kScanTotals + 4 * threadIdx.x;
  uint64_t base = sums[blockIdx.x];
  uint32_t v[4];
  uint64_t st = scan_totals(ttot, i, total_tiles, v, s_w, base);
  if (hdr->count > cap) v[0] = v[1] = v[2] = v[3] = 0u, st = 0;
  put_ranges(ranges, i, total_tiles, st, v);
}

// One tile's Gaussians of `groups` groups (column and row masks and indices `stride`
// words apart) from values[p] on; returns the place after them.  Two Gaussians per
// step and the next group's masks ahead: the loads of the indices and masks, not the
// stores, are what the loop waits for (12 frames of 120k Gaussians at 16x16 tiles:
// 129 -> 112 us).
__device__ __forceinline__ uint32_t scatter_tile(const uint32_t* col, const uint32_t* row,
                                                 const uint32_t* ids, int stride, int groups,
                                                 uint32_t* __restrict__ values, uint32_t p,
                                                 uint32_t cap) {
  uint32_t next = groups > 0 ? *col & *row : 0u;
  for (int g = 0; g < groups; ++g, ids += stride) {
    uint32_t bits = next;
    if (g + 1 < groups) {
      col += stride;
      row += stride;
      next = *col & *row;
    }
    while (bits) {
      const int k0 = __ffs(bits) - 1;
      bits &= bits - 1;
      const bool two = bits != 0;
      const int k1 = two ? __ffs(bits) - 1 : k0;
      bits &= bits - 1;  // (0 stays 0)
      const uint32_t i0 = ids[k0], i1 = ids[k1];
      if (p < cap) values[p] = i0;  // always, unless a sort wait timed out
      if (two && p + 1 < cap) values[p + 1] = i1;
      p += two ? 2 : 1;
    }
  }
  return p;
}

__global__ void __launch_bounds__(kBinThreads)
    tile_scatter_kernel(const uint32_t* __restrict__ sorted_ids, const uint2* __restrict__ srect,
                        const Header* __restrict__ hdr, const uint32_t* __restrict__ tcnt,
                        const uint2* __restrict__ ranges, uint32_t* __restrict__ values,
                        ChunkArgs a, int64_t cap) {
  grid_begin();
  extern __shared__ uint32_t smem[];
  const int b = blockIdx.y, c0 = blockIdx.x * a.per_cta, vis = (int)hdr->vis[b];
  const int r0 = c0 * a.chunk, r1 = min(r0 + a.per_cta * a.chunk, vis);
  if (r0 >= r1 || hdr->count > cap) return;
  const int words = mask_words(a.tiles_x, a.tiles_y), per = a.chunk / 32, stride = words + 32;
  const int groups = (r1 - r0 + 31) / 32, chunks = (r1 - r0 + a.chunk - 1) / a.chunk;
  grid_masks(smem, stride, srect + (size_t)b * a.N, sorted_ids + (size_t)b * a.N, r0, r1, groups,
             a.tiles_x, words);
  const uint32_t* rows = tcnt + ((size_t)b * a.n_chunk + c0) * a.NT;
  const uint2* range = ranges + (size_t)b * a.NT;
  for (int i = threadIdx.x; i < chunks * a.NT; i += kBinThreads) {
    const int c = i / a.NT, t = i - c * a.NT;
    const int ty = t / a.tiles_x, tx = t - ty * a.tiles_x;
    const uint32_t* m = smem + (size_t)c * per * stride;
    scatter_tile(m + tx, m + a.tiles_x + ty, m + words, stride, min(per, groups - c * per), values,
                 rows[i] + range[t].x, (uint32_t)cap);
  }
}

template <int W>
__global__ void __launch_bounds__(kBinThreads)
    block_scatter_kernel(const uint32_t* __restrict__ sorted_ids, const uint2* __restrict__ srect,
                         const Header* __restrict__ hdr, const uint32_t* __restrict__ tcnt,
                         const uint2* __restrict__ ranges, uint32_t* __restrict__ values,
                         ChunkArgs a, int64_t cap) {
  grid_begin();
  __shared__ uint32_t s_group[kBlockBatch * 3];
  __shared__ int s_cnt[kBinThreads / 32];
  const int b = blockIdx.y, c = blockIdx.x / a.n_block, vis = (int)hdr->vis[b];
  const int r0 = c * a.chunk, r1 = min(r0 + a.chunk, vis);
  if (r0 >= r1 || hdr->count > cap) return;
  const TileBlock t = tile_block(blockIdx.x - c * a.n_block, a);
  const OwnTiles<W> own(t, a.tiles_x);
  const uint32_t* rows = tcnt + ((size_t)b * a.n_chunk + c) * a.NT;
  const uint2* range = ranges + (size_t)b * a.NT;
  uint32_t p[W * W];
#pragma unroll
  for (int k = 0; k < W * W; ++k)
    p[k] = k < own.n ? rows[own.tile[k]] + range[own.tile[k]].x : 0u;
  const uint2* rc = srect + (size_t)b * a.N;
  const uint32_t* ids = sorted_ids + (size_t)b * a.N;
  BlockBatch<96> in;
  in.load(rc, ids, r0, r1);
  for (int base = r0; base < r1; base += kBlockBatch) {
    const int groups = block_masks<W, 96>(s_group, s_cnt, in, rc, ids, base, r1, t);
#pragma unroll
    for (int k = 0; k < W * W; ++k) {
      if (k >= own.n) break;
      p[k] = scatter_tile(s_group + own.tx[k], s_group + t.w + own.ty[k], s_group + 64, 96, groups,
                          values, p[k], (uint32_t)cap);
    }
  }
}

__global__ void export_keys_kernel(const uint2* __restrict__ ranges,
                                   const uint32_t* __restrict__ values,
                                   const uint32_t* __restrict__ zkey,
                                   uint64_t* __restrict__ keys, int N, int NT) {
  grid_begin();
  const int t = blockIdx.x, b = blockIdx.y;
  const uint2 r = ranges[(size_t)b * NT + t];
  const uint64_t hi = ((uint64_t)b * NT + t) << 32;
  for (uint32_t i = r.x + threadIdx.x; i < r.y; i += blockDim.x)
    keys[i] = hi | zkey[(size_t)b * N + values[i]];
}

}  // namespace

// look-back region: 64 words of per-pass tile counters, then one status word
// per (pass, frame, tile, digit)
constexpr size_t kLbCounters = 64;
constexpr int kMaxScanSteps = 3;  // of the column scan's last CTA; beyond, tile_range_kernel
size_t lb_bytes(const Layout& L) {
  return (kLbCounters + (size_t)4 * L.B * (L.n_dblk > 0 ? L.n_dblk : 1) * 256) * 4;
}

void launch_footprints(const Layout& L, const float* u, const float* v,
                       const int32_t* radius, const float* z,
                       unsigned char* ws, cudaStream_t st) {
  if (L.N == 0) return;
  dim3 grid((L.N + 255) / 256, L.B);
  launch(footprint_kernel, grid, 256, 0, st,
      u, v, radius, z, at<Header>(ws, L.off_header), at<uint2>(ws, L.off_rect),
      at<uint32_t>(ws, L.off_zkey), L.N, L.TW, L.TH, L.tiles_x, L.tiles_y);
  count_launches(1);
}

void launch_footprint_bound(const Layout& L, const int32_t* radius, int64_t* bound,
                            cudaStream_t st) {
  const int64_t n = (int64_t)L.B * L.N;
  if (n == 0) return;
  const int blocks = (int)min((n + 1023) / 1024, (int64_t)(4 * sm_count()));
  launch(footprint_bound_kernel, blocks, 256, 0, st, radius, n, L.TW, L.TH,
         reinterpret_cast<unsigned long long*>(bound));
  count_launches(1);
}

void launch_binning(const Layout& L, unsigned char* ws, cudaStream_t st) {
  auto* hdr = at<Header>(ws, L.off_header);
  auto* zkey = at<uint32_t>(ws, L.off_zkey);
  auto* k0 = at<uint32_t>(ws, L.off_zkey2);
  auto* k1 = k0 + (size_t)L.B * L.N;
  auto* i0 = at<uint32_t>(ws, L.off_ids);
  auto* i1 = at<uint32_t>(ws, L.off_ids2);
  auto* lb = at<uint32_t>(ws, L.off_dhist);     // pass tile counters, then status words
  auto* ghist = at<uint32_t>(ws, L.off_dtot);   // [frame][pass][digit] totals -> bases
  auto* rect = at<const uint2>(ws, L.off_rect);
  auto* srect = at<uint2>(ws, L.off_srect);
  auto* tcnt = at<uint32_t>(ws, L.off_tcnt);
  auto* ttot = at<uint32_t>(ws, L.off_ttot);
  auto* ranges = at<uint2>(ws, L.off_ranges);
  auto* values = at<uint32_t>(ws, L.off_values);
  const uint32_t* sorted = i1;
  if (L.N == 0) {
    cudaMemsetAsync(ranges, 0, (size_t)L.B * L.NT * sizeof(uint2), st);
    return;
  }
  // 1. depth sort: zkey -> (k0,i0) -> (k1,i1) -> (k0,i0) -> (k1,i1); the
  // digit totals of all passes, then one look-back kernel per pass
  const uint32_t* kin = zkey;
  const uint32_t* iin = nullptr;
  uint32_t* kout[2] = {k0, k1};
  uint32_t* iout[2] = {i0, i1};
  // the look-back words and the digit totals are adjacent: one memset
  cudaMemsetAsync(lb, 0, L.off_dtot + (size_t)L.B * 1024 * 4 - L.off_dhist, st);
  launch(dsort_hist_kernel, dim3(L.n_dblk, L.B), kSortThreads, 0, st, zkey, L.N, ghist);
  launch(dsort_bases_kernel, L.B * 4, 256, 0, st, ghist);
  for (int pass = 0; pass < 4; ++pass) {
    launch(dsort_pass_kernel, L.B * L.n_dblk, kSortThreads, 0, st,
        kin, iin, kout[pass & 1], iout[pass & 1], L.N, L.B, pass, L.n_dblk, ghist,
        lb + kLbCounters, lb + pass, hdr, pass == 3 ? rect : nullptr,
        pass == 3 ? srect : nullptr);
    kin = kout[pass & 1];
    iin = iout[pass & 1];
  }
  // 2.-3. per-chunk tile counts; per-frame column scan, totals and tile ranges;
  // 4. stable scatter
  const ChunkArgs a{L.N,  L.NT, L.tiles_x, L.tiles_y,  L.chunk,  L.n_chunk, L.chunks_per_cta,
                    L.bw, L.bh, L.blocks_x, L.n_block};
  const dim3 col_ctas((L.NT + 31) / 32, L.B);
  int launches = 9;
  if (L.n_block > 0) {
    const dim3 ctas(L.n_chunk * L.n_block, L.B);
    const bool wide = L.bw + L.bh > 32;
    const int tiles = L.B * L.NT, runs = (tiles + kScanTotals - 1) / kScanTotals;
    // (over the sort's look-back words: 4 KB per frame and more, 8 bytes per 4096 tiles)
    uint64_t* sums = runs > kMaxScanSteps ? reinterpret_cast<uint64_t*>(lb) : nullptr;
    launch(wide ? block_count_kernel<2> : block_count_kernel<1>, ctas, kBinThreads, 0, st, srect,
           hdr, tcnt, sums, sums ? runs : 0, a);
    if (!sums) {
      launch(tile_colscan_kernel<kColWarps>, col_ctas, 32 * kColWarps, 0, st, tcnt, ttot, ranges,
             sums, hdr, a, L.cap);
    } else {
      launch(tile_colscan_kernel<kColWarpsMany>, col_ctas, 32 * kColWarpsMany, 0, st, tcnt, ttot,
             ranges, sums, hdr, a, L.cap);
      launch(tile_range_kernel, runs, 32 * kColWarps, 0, st, ttot, sums, hdr, ranges, tiles, L.cap);
      ++launches;
    }
    launch(wide ? block_scatter_kernel<2> : block_scatter_kernel<1>, ctas, kBinThreads, 0, st,
           sorted, srect, hdr, tcnt, ranges, values, a, L.cap);
  } else {
    // (at most 64 groups of at most 96 words and 32 indices: 32 KB)
    const int stride = mask_words(L.tiles_x, L.tiles_y) + 32;  // words per group, with indices
    const size_t smem = (size_t)L.chunks_per_cta * (L.chunk / 32) * stride * 4;
    const dim3 ctas((L.n_chunk + L.chunks_per_cta - 1) / L.chunks_per_cta, L.B);
    launch(tile_count_kernel, ctas, kBinThreads, smem, st, srect, hdr, tcnt, a);
    launch(tile_colscan_kernel<kColWarps>, col_ctas, 32 * kColWarps, 0, st, tcnt, ttot, ranges,
           nullptr, hdr, a, L.cap);
    launch(tile_scatter_kernel, ctas, kBinThreads, smem, st, sorted, srect, hdr, tcnt, ranges,
           values, a, L.cap);
  }
  count_launches(launches);
}

void launch_export_keys(const Layout& L, uint64_t* keys, unsigned char* ws,
                        cudaStream_t st) {
  dim3 g(L.NT, L.B);
  launch(export_keys_kernel, g, 128, 0, st,
      at<const uint2>(ws, L.off_ranges), at<const uint32_t>(ws, L.off_values),
      at<const uint32_t>(ws, L.off_zkey), keys, L.N, L.NT);
  count_launches(1);
}

}  // namespace gftorf

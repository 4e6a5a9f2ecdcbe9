// k_bin.cu -- depth ordering per tile (Eq. 4: faces are composited in depth order).
//
//  1. per tile, the number of (view, face) pairs whose tile rectangle covers it.  When every
//     view's tiles fit in shared memory (TS_BIN_MAX_TILES), one block per (block of faces, view)
//     counts its pairs per tile there and writes a row of a [face block][tile] count matrix; else
//     global atomic counts per tile;
//  2. an exclusive scan of the counts (two-level: groups of 32 tiles, each tile's column of the
//     matrix summed on the way, or 4096 counts) gives each tile's segment [start, end) of the pair
//     list -- and with the matrix each block's first place in it -- the pair total and the capacity
//     check;
//  3. each pair is placed in its tile's segment (shared-memory atomics on the block's places, or
//     global atomic cursors) as the 64-bit key (float bits of the depth key << 32 | face id),
//     unique within a tile;
//  4. each segment is sorted by that key (one warp's registers up to 512 pairs, one CTA beyond: runs
//     of 128 sorted in registers, then merged in shared memory), and written out as the pair list:
//     key (global tile id << 32 | depth bits) and face id, ascending depth with ties in ascending
//     face id -- the order a stable sort of the (view, face)-ordered pairs by (tile, depth) gives.
// Every kernel reads the pair count from the device, so nothing here synchronises the host.
#include <algorithm>

#include "ts_internal.cuh"

namespace {

constexpr int SCAN_T = 1024;
constexpr int SCAN_PER = TS_SCAN_ITEMS / SCAN_T;  // 4

__device__ __forceinline__ uint32_t warp_incl_scan(uint32_t x) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
    if (lane >= o) x += y;
  }
  return x;
}

// Exclusive block scan of one value per thread (1024 threads); returns the block total in *tot.
__device__ __forceinline__ uint32_t block_excl_scan(uint32_t x, uint32_t* sm, uint32_t* tot) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const uint32_t inc = warp_incl_scan(x);
  if (lane == 31) sm[warp] = inc;
  __syncthreads();
  if (warp == 0) {
    const uint32_t w = sm[lane];
    const uint32_t wi = warp_incl_scan(w);
    sm[lane] = wi - w;
    if (lane == 31) sm[32] = wi;
  }
  __syncthreads();
  const uint32_t r = sm[warp] + inc - x;
  *tot = sm[32];
  __syncthreads();
  return r;
}

// What a group's 64-bit pair total leaves out of its 32-bit sum, for the total that k_scan_bsums forms: the
// places past 2^32 wrap, but the pair count and with it the capacity check see every pair.
__device__ __forceinline__ void keep_wraps(unsigned long long total, unsigned int* wraps) {
  const unsigned int w = (unsigned int)(total >> 32);
  if (w) atomicAdd(wraps, w);
}

__global__ void __launch_bounds__(SCAN_T) k_scan_reduce(const uint32_t* __restrict__ in, long long n,
                                                        uint32_t* __restrict__ bsums, unsigned int* wraps) {
  __shared__ unsigned long long wsum[SCAN_T / 32];
  const long long base = (long long)blockIdx.x * TS_SCAN_ITEMS;
  if (base >= n) return;
  unsigned long long s = 0;
#pragma unroll
  for (int k = 0; k < SCAN_PER; ++k) {
    const long long i = base + (long long)k * SCAN_T + threadIdx.x;
    if (i < n) s += in[i];
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  if ((threadIdx.x & 31) == 0) wsum[threadIdx.x >> 5] = s;
  __syncthreads();
  if (threadIdx.x == 0) {
    unsigned long long tot = 0;
    for (int w = 0; w < SCAN_T / 32; ++w) tot += wsum[w];
    bsums[blockIdx.x] = (uint32_t)tot;
    keep_wraps(tot, wraps);
  }
}

// Exclusive scan of the block sums in place (one block); writes the grand total, takes up *wraps (and zeroes
// it), and zeroes *zero_out (the sort's count of long lists) for the launches that follow.
__global__ void __launch_bounds__(SCAN_T) k_scan_bsums(uint32_t* bsums, long long nb, unsigned long long* total_out,
                                                       unsigned int* err, long long cap, unsigned int* wraps,
                                                       unsigned int* zero_out) {
  __shared__ uint32_t sm[33];
  __shared__ unsigned long long wsum[SCAN_T / 32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const long long per = (nb + SCAN_T - 1) / SCAN_T;
  const long long b0 = (long long)threadIdx.x * per;
  unsigned long long s = 0;
  for (long long i = b0; i < b0 + per && i < nb; ++i) s += bsums[i];
  uint32_t tot;
  uint32_t run = block_excl_scan((uint32_t)s, sm, &tot);
  // the 64-bit total guards against overflow of the 32-bit running offsets: a warp reduction,
  // then the warps' sums in order
  unsigned long long ws = s;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) ws += __shfl_xor_sync(0xffffffffu, ws, o);
  if (lane == 0) wsum[warp] = ws;
  for (long long i = b0; i < b0 + per && i < nb; ++i) {
    const uint32_t v = bsums[i];
    bsums[i] = run;
    run += v;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    unsigned long long tot64 = (unsigned long long)*wraps << 32;
    for (int w = 0; w < SCAN_T / 32; ++w) tot64 += wsum[w];
    *wraps = 0u;
    *total_out = tot64;
    if ((long long)tot64 > cap) atomicOr(err, TS_ERRBIT_CAPACITY);
    *zero_out = 0u;
  }
}

// ---------------------------------------------------------------------------- tile segments
struct TileArgs {
  const uint32_t* count;
  const short4* rect;
  const uint32_t* zbits;
  const TsView* views;
  long long VM, M, cap, n_tiles;
  uint32_t* tcnt;                  // per tile: pair count (step 1)
  uint2* ranges;                   // per tile: [start, cursor) (steps 2-3), then [start, end)
  unsigned long long* seg;         // the segments' unsorted keys (cap entries)
  unsigned int* err;
};

// Step 1: one thread per (view, face); a face adds one to each tile of its rectangle.
__global__ void __launch_bounds__(256) k_tile_count(TileArgs a) {
  const long long idx = (long long)blockIdx.x * 256 + threadIdx.x;
  if (idx >= a.VM || a.count[idx] == 0) return;
  const int view = (int)(idx / a.M);
  const TsView& vw = a.views[view];
  const short4 r = a.rect[idx];
  for (int ty = r.y; ty <= r.w; ++ty) {
    const long long trow = vw.tile_off + (long long)ty * vw.TX;
    for (int tx = r.x; tx <= r.z; ++tx) atomicAdd(a.tcnt + trow + tx, 1u);
  }
}

// Step 2, second level: the exclusive scan of the counts, written as empty ranges [start, start).
__global__ void __launch_bounds__(SCAN_T) k_tile_starts(TileArgs a, const uint32_t* __restrict__ bsums) {
  __shared__ uint32_t sm[33];
  const long long n = a.n_tiles;
  const long long base = (long long)blockIdx.x * TS_SCAN_ITEMS;
  if (base >= n) return;
  const long long i0 = base + (long long)threadIdx.x * SCAN_PER;
  uint32_t c[SCAN_PER];
  uint32_t s = 0;
#pragma unroll
  for (int k = 0; k < SCAN_PER; ++k) {
    c[k] = (i0 + k < n) ? a.tcnt[i0 + k] : 0u;
    s += c[k];
  }
  uint32_t tot;
  uint32_t off = block_excl_scan(s, sm, &tot) + bsums[blockIdx.x];
#pragma unroll
  for (int k = 0; k < SCAN_PER; ++k) {
    if (i0 + k < n) a.ranges[i0 + k] = make_uint2(off, off);
    off += c[k];
  }
}

// Step 3: one thread per (view, face); each of its tiles takes the next place of its segment.
// The places of up to four tiles are requested together (independent atomics in flight at
// once), and only then written.
__global__ void __launch_bounds__(256) k_tile_scatter(TileArgs a) {
  const long long idx = (long long)blockIdx.x * 256 + threadIdx.x;
  if (idx >= a.VM || a.count[idx] == 0) return;
  const int view = (int)(idx / a.M);
  const uint32_t face = (uint32_t)(idx - (long long)view * a.M);
  const TsView& vw = a.views[view];
  const short4 r = a.rect[idx];
  const unsigned long long key = ((unsigned long long)a.zbits[idx] << 32) | face;
  const int w = r.z - r.x + 1, h = r.w - r.y + 1;
  const long long t0 = vw.tile_off + (long long)r.y * vw.TX + r.x;
  if (w * h <= 4) {
    uint32_t pos[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const int dy = k / w, dx = k - dy * w;  // w >= 1
      if (k < w * h) pos[k] = atomicAdd(&a.ranges[t0 + (long long)dy * vw.TX + dx].y, 1u);
    }
#pragma unroll
    for (int k = 0; k < 4; ++k)
      if (k < w * h && (long long)pos[k] < a.cap) a.seg[pos[k]] = key;  // beyond: capacity bit latched
    return;
  }
  for (int ty = r.y; ty <= r.w; ++ty) {
    const long long trow = vw.tile_off + (long long)ty * vw.TX;
    for (int tx = r.x; tx <= r.z; ++tx) {
      const uint32_t pos = atomicAdd(&a.ranges[trow + tx].y, 1u);
      if ((long long)pos < a.cap) a.seg[pos] = key;
    }
  }
}

// Steps 1-3 when every view's tiles fit in shared memory: one block per (block of faces, view) counts its
// pairs per tile in shared memory, the exclusive scan of the [face block][tile] count matrix down its
// columns gives each block its first place in every tile's segment, and the block then places its pairs with
// shared-memory atomics.
//
// A warp numbers the (face, tile) pairs of 32 faces (a scan of their rectangles' sizes) and takes 32 of them
// at a time, one per lane; rectangles above WIDE_MIN tiles are queued for the whole block.  With a thread
// walking its own face's tiles, the few faces right before a camera, which cover the image, each held one
// thread for thousands of dependent steps and the launch waited for it (3 % of its issue slots used).  And
// the matrix was [tile][face block], written and read 4 bytes at a time.  Counts, scans and places together:
// 246 -> 103 us for 20 views of 300k faces (places alone 167 -> 53), 115 -> 40 for 8 views of 640x480,
// 238 -> 158 for the 12-view window of 1M faces, 275 -> 222 for 9 views of 2M.
struct MatArgs {
  const short4* rect;
  const uint32_t* zbits;
  const TsView* views;
  long long M, n_tiles, cap;
  int faces;             // per block, a multiple of BIN_T
  uint32_t* mat;         // [face block][tile]: pair counts, then their exclusive sums down the column
  const uint32_t* tpre;  // per tile: the pairs of the tiles before it in its group of 2^shift
  const uint32_t* gsum;  // per group: the pairs of the groups before it
  int shift;
  unsigned long long* seg;
};

constexpr int BIN_T = 512;
constexpr int WIDE_MIN = 128;  // tiles above which a rectangle is queued
constexpr int WIDE_MAX = 256;  // queue entries; the warps take the rectangles beyond it themselves
static_assert(TS_BIN_FACES % 1024 == 0 && 1024 % BIN_T == 0, "whole rounds of faces per thread");

struct WideFaces {
  short4 rect[WIDE_MAX];
  uint32_t z[WIDE_MAX], id[WIDE_MAX];
  unsigned n;
};

// k / w for 0 <= k < 2^20 and 1 <= w: (k + 1/2) / w lies at least 1 / (2 w) from every whole number, and the
// approximation is off by less than 2^-21 of it.
__device__ __forceinline__ int small_div(int k, int w) {
  return (int)(((float)k + 0.5f) * ts_rcp_approx((float)w));
}

// Every thread of the block calls it: put(tile of the view, depth bits, face) for each pair of the block's
// faces.  WITH_Z: the depth keys are loaded (else zero).
template <bool WITH_Z, class Put>
__device__ __forceinline__ void for_each_pair(const MatArgs& a, int v, long long blk, int TX, WideFaces& wide,
                                              Put put) {
  const int lane = threadIdx.x & 31;
  const long long vbase = (long long)v * a.M;
  const long long m0 = blk * a.faces + threadIdx.x;
  const int rounds = a.faces / BIN_T;
  const short4 none = make_short4(-1, -1, -1, -1);
  auto rect_at = [&](int k) {
    const long long m = m0 + (long long)k * BIN_T;
    return k < rounds && m < a.M ? a.rect[vbase + m] : none;
  };
  auto z_at = [&](int k) {
    const long long m = m0 + (long long)k * BIN_T;
    return WITH_Z && k < rounds && m < a.M ? a.zbits[vbase + m] : 0u;
  };
  // two rounds' loads in flight while one is worked on
  short4 r = rect_at(0), r1 = rect_at(1);
  uint32_t z = z_at(0), z1 = z_at(1);
#pragma unroll 1
  for (int k = 0; k < rounds; ++k) {
    const short4 r2 = rect_at(k + 2);
    const uint32_t z2 = z_at(k + 2);
    const uint32_t id = (uint32_t)(m0 + (long long)k * BIN_T);
    const int w = r.z - r.x + 1;
    int n = r.x >= 0 ? w * (r.w - r.y + 1) : 0;  // an invisible face's rectangle is -1
    if (n > WIDE_MIN) {
      const unsigned q = atomicAdd(&wide.n, 1u);
      if (q < WIDE_MAX) {
        wide.rect[q] = r;
        wide.z[q] = z;
        wide.id[q] = id;
        n = 0;
      }
    }
    const int corner = (int)r.y * TX + (int)r.x;
    const int total = (int)__reduce_add_sync(0xffffffffu, (unsigned)n);
    if constexpr (!WITH_Z) {
      // rectangles of a few tiles each: every lane walks its own (about a third of a numbered step's instructions a
      // tile).  50k faces of 100 views of 320 x 240: 34 us numbered, 27 so; the places, whose steps wait for an atomic's
      // answer and a store, are faster numbered (77 and 80 us at 12 views of 1M faces).
      const int most = (int)__reduce_max_sync(0xffffffffu, (unsigned)n);
      if (most <= 1 + 3 * ((total + 31) >> 5)) {
        for (int p = 0, x = 0, t = corner; p < most; ++p, ++t) {
          if (p < n) put(t, 0u, id);
          if (++x == w) {
            x = 0;
            t += TX - w;
          }
        }
        r = r1;
        r1 = r2;
        continue;
      }
    }
    const int excl = (int)warp_incl_scan((uint32_t)n) - n;
    for (int e0 = 0; e0 < total; e0 += 32) {
      const int e = e0 + lane;
      int ow = 0;  // the pair's lane: the last whose first number is at most e
#pragma unroll
      for (int s = 16; s > 0; s >>= 1)
        if (__shfl_sync(0xffffffffu, excl, ow + s) <= e) ow += s;
      const int p = e - __shfl_sync(0xffffffffu, excl, ow);
      const int pw = __shfl_sync(0xffffffffu, w, ow);
      const int pc = __shfl_sync(0xffffffffu, corner, ow);
      const uint32_t pz = WITH_Z ? __shfl_sync(0xffffffffu, z, ow) : 0u;
      const int dy = small_div(p, pw);
      if (e < total) put(pc + dy * (TX - pw) + p, pz, id - (uint32_t)lane + (uint32_t)ow);
    }
    r = r1;
    r1 = r2;
    z = z1;
    z1 = z2;
  }
  __syncthreads();
  const int nw = (int)min(wide.n, (unsigned)WIDE_MAX);
  for (int q = 0; q < nw; ++q) {
    const short4 r = wide.rect[q];
    const int w = r.z - r.x + 1, n = w * (r.w - r.y + 1);
    for (int p = threadIdx.x; p < n; p += BIN_T) {
      const int dy = small_div(p, w);
      put((r.y + dy) * TX + r.x + (p - dy * w), wide.z[q], wide.id[q]);
    }
  }
}

__global__ void __launch_bounds__(BIN_T, 3) k_bin_counts(MatArgs a) {
  extern __shared__ uint32_t hcnt[];
  __shared__ WideFaces wide;
  const int v = blockIdx.y;
  const TsView& vw = a.views[v];
  const int TX = vw.TX, T = TX * vw.TY;
  if (threadIdx.x == 0) wide.n = 0u;
  for (int t = threadIdx.x; t < T; t += BIN_T) hcnt[t] = 0u;
  __syncthreads();
  for_each_pair<false>(a, v, blockIdx.x, TX, wide, [&](int t, uint32_t, uint32_t) { atomicAdd(&hcnt[t], 1u); });
  __syncthreads();
  uint32_t* row = a.mat + (long long)blockIdx.x * a.n_tiles + vw.tile_off;
  for (int t = threadIdx.x; t < T; t += BIN_T) row[t] = hcnt[t];
}

// The exclusive sums down each tile's column in place; the tiles' totals, scanned within the group, and the
// group's total.  One block per 32 tiles, a lane per tile and a warp per share of the rows, up to 64 rows at a
// time in registers; for many tiles of at most TS_BIN_FEW rows one block per 256 tiles, a thread per tile, so that
// views of many tiles and few faces do not launch a block of mostly idle warps per 32 tiles, nor scan as many groups:
// 16 views of 1920 x 1080 at 8 x 8 tiles, 2000 faces, columns and scan 46 -> 11 us.
constexpr int COL_WARPS = 8, COL_ROWS = 8;  // warps per block, most rows per warp at a time
__global__ void __launch_bounds__(32 * COL_WARPS) k_bin_columns(uint32_t* __restrict__ mat, long long n_tiles, int B,
                                                                 uint32_t* __restrict__ tpre,
                                                                 uint32_t* __restrict__ gsum, unsigned int* wraps) {
  __shared__ uint32_t part[COL_WARPS][32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const long long t = (long long)blockIdx.x * 32 + lane;
  const bool in = t < n_tiles;
  uint32_t carry = 0u;
  for (int r0 = 0; r0 < B; r0 += COL_WARPS * COL_ROWS) {
    const int left = min(B - r0, COL_WARPS * COL_ROWS), per = (left + COL_WARPS - 1) / COL_WARPS;
    const int k1 = min(per, left - warp * per);  // this warp's rows: r0 + warp * per + [0, k1)
    uint32_t* col = mat + (long long)(r0 + warp * per) * n_tiles + t;
    uint32_t c[COL_ROWS], s = 0u;
#pragma unroll
    for (int k = 0; k < COL_ROWS; ++k) {
      c[k] = in && k < k1 ? col[(long long)k * n_tiles] : 0u;
      s += c[k];
    }
    part[warp][lane] = s;
    __syncthreads();
    uint32_t off = carry;
#pragma unroll
    for (int w = 0; w < COL_WARPS; ++w) {
      const uint32_t x = part[w][lane];
      carry += x;
      off += w < warp ? x : 0u;
    }
    __syncthreads();
#pragma unroll
    for (int k = 0; k < COL_ROWS; ++k) {
      if (in && k < k1) col[(long long)k * n_tiles] = off;
      off += c[k];
    }
  }
  if (warp == 0) {
    const uint32_t incl = warp_incl_scan(carry);
    if (in) tpre[t] = incl - carry;
    // the group's total in 64 bits (a tile's is below 2^31): 32 tiles of 2^27 faces each pass 2^32
    const unsigned long long tot = ((unsigned long long)__reduce_add_sync(0xffffffffu, carry >> 16) << 16) +
                                   __reduce_add_sync(0xffffffffu, carry & 0xffffu);
    if (lane == 31) {
      gsum[blockIdx.x] = incl;
      keep_wraps(tot, wraps);
    }
  }
}

__global__ void __launch_bounds__(256) k_bin_columns_few(uint32_t* __restrict__ mat, long long n_tiles, int B,
                                                         uint32_t* __restrict__ tpre, uint32_t* __restrict__ gsum) {
  static_assert(256ll * TS_BIN_FEW * TS_BIN_FACES < (1ll << 32), "a group's pairs fit 32 bits");
  __shared__ uint32_t wsum[8];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const long long t = (long long)blockIdx.x * 256 + threadIdx.x;
  uint32_t c[TS_BIN_FEW], total = 0u;
#pragma unroll
  for (int k = 0; k < TS_BIN_FEW; ++k) c[k] = t < n_tiles && k < B ? mat[k * n_tiles + t] : 0u;
#pragma unroll
  for (int k = 0; k < TS_BIN_FEW; ++k) {
    if (t < n_tiles && k < B) mat[k * n_tiles + t] = total;
    total += c[k];
  }
  const uint32_t incl = warp_incl_scan(total);
  if (lane == 31) wsum[warp] = incl;
  __syncthreads();
  uint32_t before = 0u, all = 0u;
#pragma unroll
  for (int w = 0; w < 8; ++w) {
    before += w < warp ? wsum[w] : 0u;
    all += wsum[w];
  }
  if (t < n_tiles) tpre[t] = before + incl - total;
  if (threadIdx.x == 0) gsum[blockIdx.x] = all;
}

__global__ void __launch_bounds__(BIN_T, 3) k_bin_place(MatArgs a) {
  extern __shared__ uint32_t place[];
  __shared__ WideFaces wide;
  const int v = blockIdx.y;
  const TsView& vw = a.views[v];
  const int TX = vw.TX, T = TX * vw.TY;
  if (threadIdx.x == 0) wide.n = 0u;
  const uint32_t* row = a.mat + (long long)blockIdx.x * a.n_tiles;
  for (int t = threadIdx.x; t < T; t += BIN_T) {
    const long long g = vw.tile_off + t;
    // (a group of 32 or 256 tiles; a shift by a register leaves 32 registers for 36 and so four blocks on a
    // multiprocessor for three: 62 us for 53 at 20 views of 300k faces, 69 for 77 at 12 of 1M)
    place[t] = row[g] + a.tpre[g] + (a.shift == 5 ? a.gsum[g / 32] : a.gsum[g / 256]);
  }
  __syncthreads();
  for_each_pair<true>(a, v, blockIdx.x, TX, wide, [&](int t, uint32_t z, uint32_t id) {
    const uint32_t pos = atomicAdd(&place[t], 1u);
    // beyond: the scan has latched the capacity bit
    if ((long long)pos < a.cap) a.seg[pos] = ((unsigned long long)z << 32) | id;
  });
}

// Step 4.  In registers, bitonic networks in the form whose every compare-exchange moves the smaller key to
// the lower index (each merge starts by comparing mirrored positions); positions past a segment's end
// hold +infinity and stay behind its keys.
struct SortOut {
  const unsigned long long* seg;
  unsigned long long* keys;
  uint32_t* vals;
  uint2* ranges;           // cut to the capacity here
  long long n_tiles, cap;
  uint32_t* large;         // tiles left to the CTA-wide sort
  unsigned int* n_large;
  const uint32_t* tpre;    // with the count matrix: pairs of the tiles before this one in its group, else null
  const uint32_t* gsum;    // (ranges from the scatter); pairs of the groups before
  int shift;               // log2 of the tiles of a group
  const unsigned long long* n_pairs;
};

__device__ __forceinline__ void put_pair(const SortOut& o, long long t, long long pos, unsigned long long k) {
  o.keys[pos] = ((unsigned long long)t << 32) | (k >> 32);
  o.vals[pos] = (uint32_t)k;
}

constexpr int WARP_SORT_MAX = 512;  // pairs a warp sorts in its registers (16 per lane)
constexpr int SORT_WARPS_PER_BLOCK = 8;
constexpr int SORT_TILES = 2;  // tiles a warp takes of at least SORT_TILES_FROM
constexpr long long SORT_TILES_FROM = 40000;

// Keep the smaller (lower) or the larger key of a compare-exchange with a lane that keeps the other.
__device__ __forceinline__ unsigned long long keep_key(unsigned long long x, unsigned long long y, bool lower) {
  return (y < x) == lower ? y : x;
}
__device__ __forceinline__ void cmp_exchange(unsigned long long& a, unsigned long long& b) {
  const bool sw = b < a;
  const unsigned long long lo = sw ? b : a, hi = sw ? a : b;
  a = lo;
  b = hi;
}

// Sort a warp's 32 * K keys, K per lane, so that position lane * K + r holds the ascending order.
// Exchanges at distances below K stay in the lane's registers, the others are lane shuffles: of the
// 36 steps of 256 keys 21 need no shuffle, and nothing touches shared memory or divides an index.
template <int K>
__device__ __forceinline__ void warp_sort(unsigned long long (&x)[K], int lane) {
#pragma unroll
  for (int k = 2; k <= K; k <<= 1) {  // within the lane
#pragma unroll
    for (int r = 0; r < K; ++r)
      if ((r & (k >> 1)) == 0) cmp_exchange(x[r], x[r ^ (k - 1)]);
#pragma unroll
    for (int j = k >> 2; j > 0; j >>= 1)
#pragma unroll
      for (int r = 0; r < K; ++r)
        if ((r & j) == 0) cmp_exchange(x[r], x[r ^ j]);
  }
#pragma unroll 1
  for (int kl = 2; kl <= 32; kl <<= 1) {  // merges of kl lanes' keys
    {  // mirrored positions: lane ^ (kl - 1), register K - 1 - r
      const bool lower = (lane & (kl >> 1)) == 0;
#pragma unroll
      for (int r = 0; r < K / 2; ++r) {
        const unsigned long long y0 = __shfl_xor_sync(0xffffffffu, x[K - 1 - r], kl - 1);
        const unsigned long long y1 = __shfl_xor_sync(0xffffffffu, x[r], kl - 1);
        x[r] = keep_key(x[r], y0, lower);
        x[K - 1 - r] = keep_key(x[K - 1 - r], y1, lower);
      }
    }
#pragma unroll 1
    for (int j = kl >> 2; j > 0; j >>= 1) {
      const bool lower = (lane & j) == 0;
#pragma unroll
      for (int r = 0; r < K; ++r) x[r] = keep_key(x[r], __shfl_xor_sync(0xffffffffu, x[r], j), lower);
    }
#pragma unroll
    for (int j = K >> 1; j > 0; j >>= 1)
#pragma unroll
      for (int r = 0; r < K; ++r)
        if ((r & j) == 0) cmp_exchange(x[r], x[r ^ j]);
  }
}

// Place of position p in a shared-memory key buffer: lanes that write 4, 8 or 16 consecutive keys
// each, and lanes that read consecutive ones, both hit distinct banks.
__device__ __forceinline__ int key_place(int p) { return p ^ ((p >> 4) & 15); }

// Sort a segment of 64 < n <= 32 * K pairs in the warp's registers; the sorted keys go through the
// warp's shared buffer so that the writes to memory are coalesced.
template <int K>
__device__ __forceinline__ void sort_segment(const SortOut& o, long long t, long long start, int n, int lane,
                                             unsigned long long* buf) {
  unsigned long long x[K];
#pragma unroll
  for (int r = 0; r < K; ++r) x[r] = r * 32 + lane < n ? o.seg[start + r * 32 + lane] : ~0ull;
  warp_sort<K>(x, lane);
#pragma unroll
  for (int r = 0; r < K; ++r) buf[key_place(lane * K + r)] = x[r];
  __syncwarp();
#pragma unroll
  for (int r = 0; r < K; ++r)
    if (r * 32 + lane < n) put_pair(o, t, start + r * 32 + lane, buf[key_place(r * 32 + lane)]);
  __syncwarp();  // the warp's next tile writes the buffer
}

// Sort the n >= 1 pairs of tile t, which start at `start` of the segments; lists beyond WARP_SORT_MAX are listed for
// the CTA-wide kernel.
__device__ __forceinline__ void sort_tile(const SortOut& o, long long t, long long start, int n, int lane,
                                          unsigned long long* buf) {
  if (n <= 32) {
    unsigned long long x = lane < n ? o.seg[start + lane] : ~0ull;
#pragma unroll
    for (int k = 2; k <= 32; k <<= 1) {
      {
        const unsigned long long y = __shfl_xor_sync(0xffffffffu, x, k - 1);
        const bool lower = (lane & (k >> 1)) == 0;
        x = lower ? min(x, y) : max(x, y);
      }
#pragma unroll
      for (int j = k >> 2; j > 0; j >>= 1) {
        const unsigned long long y = __shfl_xor_sync(0xffffffffu, x, j);
        const bool lower = (lane & j) == 0;
        x = lower ? min(x, y) : max(x, y);
      }
    }
    if (lane < n) put_pair(o, t, start + lane, x);
    return;
  }
  if (n <= 64) {  // two keys per lane: x0 at position lane, x1 at position 32 + lane
    unsigned long long x0 = o.seg[start + lane];
    unsigned long long x1 = 32 + lane < n ? o.seg[start + 32 + lane] : ~0ull;
#pragma unroll
    for (int k = 2; k <= 32; k <<= 1) {  // each half sorted as in the 32-key network
      {
        const unsigned long long y0 = __shfl_xor_sync(0xffffffffu, x0, k - 1);
        const unsigned long long y1 = __shfl_xor_sync(0xffffffffu, x1, k - 1);
        const bool lower = (lane & (k >> 1)) == 0;
        x0 = lower ? min(x0, y0) : max(x0, y0);
        x1 = lower ? min(x1, y1) : max(x1, y1);
      }
#pragma unroll
      for (int j = k >> 2; j > 0; j >>= 1) {
        const unsigned long long y0 = __shfl_xor_sync(0xffffffffu, x0, j);
        const unsigned long long y1 = __shfl_xor_sync(0xffffffffu, x1, j);
        const bool lower = (lane & j) == 0;
        x0 = lower ? min(x0, y0) : max(x0, y0);
        x1 = lower ? min(x1, y1) : max(x1, y1);
      }
    }
    {  // merge of 64: position lane pairs with 63 - lane, i.e. x1 of lane 31 - lane
      const unsigned long long y0 = __shfl_sync(0xffffffffu, x1, 31 - lane);
      const unsigned long long y1 = __shfl_sync(0xffffffffu, x0, 31 - lane);
      x0 = min(x0, y0);
      x1 = max(x1, y1);
    }
#pragma unroll
    for (int j = 16; j > 0; j >>= 1) {
      const unsigned long long y0 = __shfl_xor_sync(0xffffffffu, x0, j);
      const unsigned long long y1 = __shfl_xor_sync(0xffffffffu, x1, j);
      const bool lower = (lane & j) == 0;
      x0 = lower ? min(x0, y0) : max(x0, y0);
      x1 = lower ? min(x1, y1) : max(x1, y1);
    }
    put_pair(o, t, start + lane, x0);
    if (32 + lane < n) put_pair(o, t, start + 32 + lane, x1);
    return;
  }
  if (n > WARP_SORT_MAX) {
    if (lane == 0) {
      const unsigned slot = atomicAdd(o.n_large, 1u);
      if ((long long)slot < o.n_tiles) o.large[slot] = (uint32_t)t;
    }
    return;
  }
  if (n <= 128) sort_segment<4>(o, t, start, n, lane, buf);
  else if (n <= 256) sort_segment<8>(o, t, start, n, lane, buf);
  else sort_segment<16>(o, t, start, n, lane, buf);
}

// A warp takes TILES consecutive tiles, their keys in registers.  Issue-bound (about 6 warp instructions a key at 512
// keys, 4.5 at 128).  Lists of more than 64 pairs in shared memory, with an integer division per exchange, took 161 us
// where this takes 73 (12 views of a 1M-face map, 127 pairs a tile) and 35 where it takes 9 (mesh, 561k pixels).
// An empty or short list is two dependent loads and a store, and with one tile a warp such tiles wait for the 32 places
// of a multiprocessor that 64 registers leave; so from SORT_TILES_FROM tiles on a warp takes two, and the compiler's 48
// registers leave 40 places: 518k tiles of 2000 faces 93 -> 54 us, 20 views of 300k faces 76 -> 69.  (Below, two tiles
// a warp leave places empty: 57k tiles of the 12-view window 85 us either way, 117 with four.)
template <int TILES>
__global__ void __launch_bounds__(32 * SORT_WARPS_PER_BLOCK, TILES == 1 ? 4 : 5) k_tile_sort(SortOut o) {
  __shared__ unsigned long long sbuf[SORT_WARPS_PER_BLOCK][WARP_SORT_MAX];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const long long t0 = ((long long)blockIdx.x * SORT_WARPS_PER_BLOCK + warp) * TILES;
  if (t0 >= o.n_tiles) return;
  // lane i: the segment of tile t0 + i, from the scanned totals (its first place, the next tile's, the pair total
  // after the last tile), else as the scatter left it in ranges
  const long long tl = TILES == 1 ? t0 : t0 + lane;
  auto first_of = [&](long long t) {
    return t < o.n_tiles ? o.tpre[t] + o.gsum[t >> o.shift] : (uint32_t)min(*o.n_pairs, 0xffffffffull);
  };
  uint2 rg = make_uint2(0u, 0u);
  if (TILES == 1) {
    rg = o.tpre ? make_uint2(first_of(tl), first_of(tl + 1)) : o.ranges[tl];
  } else if (o.tpre) {
    rg.x = lane <= TILES ? first_of(min(tl, o.n_tiles)) : 0u;
    rg.y = __shfl_down_sync(0xffffffffu, rg.x, 1);
  } else if (lane < TILES && tl < o.n_tiles) {
    rg = o.ranges[tl];
  }
  const long long first = min((long long)rg.x, o.cap);
  const long long last = max(first, min((long long)rg.y, o.cap));  // (an end past 2^32 has wrapped to below its start)
  // the tile's range for the passes that follow; past the capacity (its bit is latched) the lists
  // are cut, and the ranges with them, so that no later pass reads outside the pair list
  const bool mine = lane < TILES && tl < o.n_tiles;
  if (mine && (o.tpre || first != rg.x || last != rg.y)) o.ranges[tl] = make_uint2((uint32_t)first, (uint32_t)last);
  const int len = (int)(last - first);
  if constexpr (TILES == 1) {
    if (len > 0) sort_tile(o, t0, first, len, lane, sbuf[warp]);
  } else {
#pragma unroll 1
    for (unsigned rem = __ballot_sync(0xffffffffu, mine && len > 0); rem; rem &= rem - 1) {
      const int i = __ffs(rem) - 1;
      sort_tile(o, t0 + i, __shfl_sync(0xffffffffu, (unsigned int)first, i), __shfl_sync(0xffffffffu, len, i), lane,
                sbuf[warp]);
    }
  }
}

constexpr int LARGE_T = 256;
constexpr int LARGE_ITEMS = 4096;  // keys sorted in shared memory at a time, in two buffers (64 KB)
constexpr int LARGE_RUN = 128;     // keys a warp sorts in registers (4 per lane) before the merges
constexpr int LARGE_VT = 8;        // consecutive outputs a thread merges

// One merge level of a block's n keys: sorted runs of w keys (w a power of two, the last one shorter)
// become runs of 2w.  A thread finds where its LARGE_VT consecutive outputs start in the two runs by
// bisection along their diagonal (merge path) and merges serially: 0.7 warp instructions a key.
template <typename I, typename Buf>  // I: the type of a position
__device__ __forceinline__ void merge_level(const Buf& src, const Buf& dst, I n, I w) {
  for (I o = (I)threadIdx.x * LARGE_VT; o < n; o += LARGE_T * LARGE_VT) {
    const I base = o & ~(2 * w - 1), d = o - base;
    const I la = min(w, n - base), lb = max((I)0, min(w, n - base - w));
    I lo = max((I)0, d - lb), hi = min(d, la);
    while (lo < hi) {
      const I mid = (lo + hi) >> 1;
      if (src.get(base + mid) < src.get(base + w + d - 1 - mid)) lo = mid + 1;
      else hi = mid;
    }
    I i = lo, j = d - lo;
    unsigned long long ka = i < la ? src.get(base + i) : ~0ull, kb = j < lb ? src.get(base + w + j) : ~0ull;
#pragma unroll
    for (int v = 0; v < LARGE_VT; ++v) {
      if (o + v >= n) break;
      const bool a = ka < kb;  // keys are unique, and below ~0 while any is left
      dst.put(o + v, a ? ka : kb);
      if (a) {
        ++i;
        ka = i < la ? src.get(base + i) : ~0ull;
      } else {
        ++j;
        kb = j < lb ? src.get(base + w + j) : ~0ull;
      }
    }
  }
}

struct SharedKeys {
  unsigned long long* p;
  __device__ __forceinline__ unsigned long long get(int i) const { return p[key_place(i)]; }
  __device__ __forceinline__ void put(int i, unsigned long long k) const { p[key_place(i)] = k; }
};
struct GlobalKeys {
  unsigned long long* p;
  __device__ __forceinline__ unsigned long long get(long long i) const { return p[i]; }
  __device__ __forceinline__ void put(long long i, unsigned long long k) const { p[i] = k; }
};

// The listed long segments, one CTA each (grid-stride over the list).  LARGE_ITEMS keys at a time are
// sorted in shared memory; a longer segment's sorted parts are then merged in global memory, between
// the segment buffer and the segment's place in the output.  (A bitonic network over the whole
// segment in shared memory took 574 us of a 9-view render of 2M faces where this takes 85, 120 us of a
// 12-view window of 1M faces where this takes 21.)
__global__ void __launch_bounds__(LARGE_T) k_tile_sort_large(SortOut o, unsigned long long* seg) {
  extern __shared__ __align__(16) unsigned long long lbuf[];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const unsigned nl = min(*o.n_large, (unsigned)o.n_tiles);
  for (unsigned e = blockIdx.x; e < nl; e += gridDim.x) {
    const long long t = o.large[e];
    const uint2 rg = o.ranges[t];  // already cut to the capacity
    const long long start = rg.x;
    const long long len = (long long)rg.y - start;
    for (long long c0 = 0; c0 < len; c0 += LARGE_ITEMS) {
      const int n = (int)min((long long)LARGE_ITEMS, len - c0);
      SharedKeys cur{lbuf}, nxt{lbuf + LARGE_ITEMS};
      for (int r0 = warp * LARGE_RUN; r0 < n; r0 += (LARGE_T / 32) * LARGE_RUN) {
        unsigned long long x[4];
#pragma unroll
        for (int r = 0; r < 4; ++r)
          x[r] = r0 + r * 32 + lane < n ? seg[start + c0 + r0 + r * 32 + lane] : ~0ull;
        warp_sort<4>(x, lane);
#pragma unroll
        for (int r = 0; r < 4; ++r)
          if (r0 + lane * 4 + r < n) cur.put(r0 + lane * 4 + r, x[r]);
      }
      __syncthreads();
      for (int w = LARGE_RUN; w < n; w <<= 1) {
        merge_level(cur, nxt, n, w);
        __syncthreads();
        const SharedKeys sw = cur;
        cur = nxt;
        nxt = sw;
      }
      if (len <= LARGE_ITEMS) {
        for (int i = threadIdx.x; i < n; i += LARGE_T) put_pair(o, t, start + i, cur.get(i));
      } else {
        for (int i = threadIdx.x; i < n; i += LARGE_T) seg[start + c0 + i] = cur.get(i);
      }
      __syncthreads();
    }
    if (len > LARGE_ITEMS) {
      GlobalKeys src{seg + start}, dst{o.keys + start};
      for (long long w = LARGE_ITEMS; w < len; w <<= 1) {
        merge_level(src, dst, len, w);
        __syncthreads();
        const GlobalKeys sw = src;
        src = dst;
        dst = sw;
      }
      for (long long i = threadIdx.x; i < len; i += LARGE_T) put_pair(o, t, start + i, src.get(i));
      __syncthreads();
    }
  }
}

}  // namespace

cudaError_t ts_launch_bin(const TsPlanImpl* p, const TsWs& w, cudaStream_t s) {
  const long long VM = (long long)p->V * p->M;
  cudaError_t e = cudaSuccess;
  if (VM == 0) {  // no records: empty ranges and no pairs (otherwise the kernels below write them)
    e = cudaMemsetAsync(w.ranges, 0, (size_t)p->n_tiles * sizeof(uint2), s);
    if (e == cudaSuccess) e = cudaMemsetAsync(&w.hdr->n_large, 0, sizeof(unsigned int), s);
    if (e == cudaSuccess) e = cudaMemsetAsync(&w.hdr->n_pairs, 0, sizeof(unsigned long long), s);
    return e;
  }
  if (p->bin_blocks > 0) {
    // 1-3 with shared-memory counts: counts, their scan (the total is the pair count; above the
    // capacity latches its bit), places, ranges
    MatArgs ma{w.rect, w.zbits, w.views, p->M, p->n_tiles, p->cap, (int)p->bin_faces, w.tmat, w.tcnt, w.bsums,
               (int)p->bin_shift, w.keys[1]};
    const int smem = (int)(p->max_view_tiles * sizeof(uint32_t));
    e = ts_smem_limit((const void*)k_bin_counts, smem);
    if (e == cudaSuccess) e = ts_smem_limit((const void*)k_bin_place, smem);
    if (e != cudaSuccess) return e;
    const dim3 grid((unsigned)p->bin_blocks, (unsigned)p->V);
    k_bin_counts<<<grid, BIN_T, smem, s>>>(ma);
    const unsigned ng = (unsigned)(((p->n_tiles - 1) >> p->bin_shift) + 1);
    if (p->bin_shift == 8)
      k_bin_columns_few<<<ng, 256, 0, s>>>(w.tmat, p->n_tiles, (int)p->bin_blocks, w.tcnt, w.bsums);
    else
      k_bin_columns<<<ng, 32 * COL_WARPS, 0, s>>>(w.tmat, p->n_tiles, (int)p->bin_blocks, w.tcnt, w.bsums,
                                                   &w.hdr->pair_wraps);
    k_scan_bsums<<<1, SCAN_T, 0, s>>>(w.bsums, ng, &w.hdr->n_pairs, &w.hdr->error_bits, p->cap,
                                       &w.hdr->pair_wraps, &w.hdr->n_large);
    k_bin_place<<<grid, BIN_T, smem, s>>>(ma);
  } else {
    // 1-3 with global counts: counts, their scan, starts, places
    e = cudaMemsetAsync(w.tcnt, 0, (size_t)p->n_tiles * sizeof(uint32_t), s);
    if (e != cudaSuccess) return e;
    TileArgs ta{w.count, w.rect, w.zbits, w.views, VM, p->M, p->cap, p->n_tiles, w.tcnt, w.ranges, w.keys[1],
                &w.hdr->error_bits};
    const unsigned nf = (unsigned)((VM + 255) / 256);
    k_tile_count<<<nf, 256, 0, s>>>(ta);
    const unsigned nb = (unsigned)((p->n_tiles + TS_SCAN_ITEMS - 1) / TS_SCAN_ITEMS);
    k_scan_reduce<<<nb, SCAN_T, 0, s>>>(w.tcnt, p->n_tiles, w.bsums, &w.hdr->pair_wraps);
    k_scan_bsums<<<1, SCAN_T, 0, s>>>(w.bsums, nb, &w.hdr->n_pairs, &w.hdr->error_bits, p->cap,
                                       &w.hdr->pair_wraps, &w.hdr->n_large);
    k_tile_starts<<<nb, SCAN_T, 0, s>>>(ta, w.bsums);
    k_tile_scatter<<<nf, 256, 0, s>>>(ta);
  }
  // 4: the segments' sorts
  // (with the matrix, the sort also writes each tile's range)
  SortOut so{w.keys[1], w.keys[0], w.vals[0], w.ranges, p->n_tiles, p->cap, w.tlarge, &w.hdr->n_large,
             p->bin_blocks > 0 ? w.tcnt : nullptr, w.bsums, (int)p->bin_shift, &w.hdr->n_pairs};
  const long long per = p->n_tiles >= SORT_TILES_FROM ? SORT_TILES : 1;
  const unsigned nw = (unsigned)((p->n_tiles + per * SORT_WARPS_PER_BLOCK - 1) / (per * SORT_WARPS_PER_BLOCK));
  if (per > 1) k_tile_sort<SORT_TILES><<<nw, 32 * SORT_WARPS_PER_BLOCK, 0, s>>>(so);
  else k_tile_sort<1><<<nw, 32 * SORT_WARPS_PER_BLOCK, 0, s>>>(so);
  constexpr int large_smem = 2 * LARGE_ITEMS * (int)sizeof(unsigned long long);
  e = ts_smem_limit((const void*)k_tile_sort_large, large_smem);
  if (e != cudaSuccess) return e;
  k_tile_sort_large<<<3u * (unsigned)ts_sm_count(), LARGE_T, large_smem, s>>>(so, w.keys[1]);  // 3 fit on an SM
  return cudaGetLastError();
}

// Index construction of Section 4: for every (repetition j, dimension f)
// the windows ordered lexicographically by their K-value hash strings, so
// that every prefix length i groups colliding windows into contiguous runs.
//
// A most-significant-digit radix partition followed by shared-memory
// sorts.  Level t (t = 0, 1, ...) partitions ranges ("items") stably by
// hash value t (one byte of the big-endian composite key); a partition
// never moves an entry out of its item, so every entry lands in its final
// position's bucket.  Buckets of at most kLocalMax entries are packed, in
// order, into chunks that one CTA then sorts completely in shared memory
// by (key, window); larger buckets become the items of level t + 1.  After level
// K - 1 every bucket holds equal keys and is already in order.  On the
// hash strings of z-normalised windows one level usually suffices: the
// largest bucket of the first hash value holds a few percent of the
// windows.
//
// Each level is three kernels: per-tile digit histograms, a per-item scan
// of (digit, tile) counts that also classifies the buckets (chunks for the
// shared-memory sort, items for the next level), and a stable scatter that
// ranks equal digits with warp match masks and writes each tile in digit
// order through shared memory.  The final kernel writes, per rank, the
// sorted window and the number of hash values shared with the previous
// rank (the longest common prefix, 0..K), which is all the traversal needs.
//
// Every kernel reads its work counts from device counters (grid-stride
// loops), so the levels can run without the host: the index build reads
// the counts after each level to size the next launch exactly, the
// allocation-free entry point launches all K levels with fixed grids.
#include "internal.h"

#include <algorithm>

namespace momenti {

namespace {

constexpr int kThreads = 256;
constexpr int kItems = 8;                      // per thread
constexpr int kTile = kSortTile;               // entries per partition tile
static_assert(kTile == kThreads * kItems, "partition tile");
constexpr int kWarps = kThreads / 32;
constexpr int kWarpSpan = kTile / kWarps;      // 256 entries per warp
constexpr int kRounds = kWarpSpan / 32;        // 8

constexpr int kLocalThreads = 256;
constexpr int kLocalBlocks = 4;                              // CTAs per SM (64 registers a thread)
constexpr int kLocalWarps = kLocalThreads / 32;
constexpr int kLocalItems = kSortLocalMax / kLocalThreads;   // 8 per thread
constexpr int kBinBits = 11;                                 // bins of a chunk: about one per entry
constexpr int kBins = 1 << kBinBits;
static_assert(kBins % kLocalThreads == 0 && kSortLocalMax <= 4096, "bin and rank travel in one word");

// counters: [2 t] items and [2 t + 1] tiles of level t (t = 0..8), then
constexpr int kCntChunks = 20;   // chunks for the shared-memory sort
constexpr int kCntOverflow = 22; // a capacity was exceeded

struct Level {
  // level 0 reads keys [j][a][f] and the implicit value a; later levels
  // read the ping-pong buffers [seg][M]
  const uint64_t* keys;
  const uint64_t* kin;
  const uint32_t* vin;
  uint64_t* kout;
  uint32_t* vout;
  int64_t M;
  int D, j0, t, K, segs;
  const SortItem* items;
  SortItem* items_next;
  const uint64_t* tile_item;
  uint64_t* tile_next;
  uint32_t* hist;
  SortChunk* chunks;
  uint32_t* cnt;
  uint32_t item_cap, tile_cap, chunk_cap;
  __device__ __forceinline__ uint64_t load_key(uint32_t seg, int64_t p) const {
    if (t == 0) {
      const int j = j0 + int(seg) / D, f = int(seg) - (int(seg) / D) * D;
      return keys[(int64_t(j) * M + p) * D + f];
    }
    return kin[int64_t(seg) * M + p];
  }
  __device__ __forceinline__ void load(uint32_t seg, int64_t p, uint64_t& k, uint32_t& v) const {
    if (t == 0) {
      k = load_key(seg, p);
      v = uint32_t(p);
    } else {
      k = kin[int64_t(seg) * M + p];
      v = vin[int64_t(seg) * M + p];
    }
  }
  __device__ __forceinline__ uint32_t digit(uint64_t k) const {
    return uint32_t(k >> (56 - 8 * t)) & 255u;
  }
  // the item of a launch tile, false for an entry that is not a valid tile of
  // a valid item (only after an overflow; nothing outside the buffers is read)
  __device__ __forceinline__ bool tile_of(uint32_t tile, SortItem& it, uint32_t& tt) const {
    const uint64_t te = tile_item[tile];
    const uint32_t ii = uint32_t(te);
    tt = uint32_t(te >> 32);
    if (ii >= min(cnt[2 * t], item_cap)) return false;
    it = items[ii];
    return it.seg < uint32_t(segs) && int64_t(it.start) + it.size <= M &&
           tt < (it.size + kTile - 1) / kTile &&
           int64_t(it.hist0) + (it.size + kTile - 1) / kTile <= int64_t(tile_cap);
  }
};

__device__ __forceinline__ uint32_t ntiles(uint32_t size) { return (size + kTile - 1) / kTile; }

// Level 0: one item per segment.
// Launch tiles run segment-fastest, so that the D segments of a repetition,
// which read the same rows of the key array, are processed together.
__global__ void k_sort_init(int segs, int64_t M, SortItem* items, uint64_t* tile_item,
                            uint32_t* cnt) {
  const uint32_t tpm = uint32_t((M + kTile - 1) / kTile);
  const int64_t total = int64_t(segs) * tpm;
  for (int64_t q = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; q < total;
       q += int64_t(gridDim.x) * blockDim.x) {
    const uint32_t seg = uint32_t(q % segs), tt = uint32_t(q / segs);
    tile_item[q] = (uint64_t(tt) << 32) | seg;
    if (tt == 0) items[seg] = SortItem{seg, 0u, uint32_t(M), seg * tpm, 0u, {0u, 0u, 0u}};
  }
  if (blockIdx.x == 0 && threadIdx.x < 32) {
    for (int c = threadIdx.x; c < 32; c += 32) cnt[c] = 0;
    __syncwarp();
    if (threadIdx.x == 0) {
      cnt[0] = uint32_t(segs);
      cnt[1] = uint32_t(total);
    }
  }
}

__global__ void __launch_bounds__(kThreads) k_sort_hist(Level lv) {
  __shared__ uint32_t h[256];
  // the next level's counts start from zero (its items are added by the
  // scan kernel of this level, which runs after this one)
  if (blockIdx.x == 0 && threadIdx.x < 2 && lv.t < 8) lv.cnt[2 * (lv.t + 1) + threadIdx.x] = 0;
  const uint32_t nt = min(lv.cnt[2 * lv.t + 1], lv.tile_cap);
  for (uint32_t tile = blockIdx.x; tile < nt; tile += gridDim.x) {
    SortItem it;
    uint32_t tt;
    if (!lv.tile_of(tile, it, tt)) continue;
    for (int d = threadIdx.x; d < 256; d += kThreads) h[d] = 0;
    __syncthreads();
    const int64_t base = int64_t(it.start) + int64_t(tt) * kTile;
    const int64_t end = int64_t(it.start) + it.size;
    uint64_t k[kItems];
#pragma unroll
    for (int r = 0; r < kItems; ++r) {
      const int64_t p = base + r * kThreads + threadIdx.x;
      k[r] = p < end ? lv.load_key(it.seg, p) : 0ull;
    }
#pragma unroll
    for (int r = 0; r < kItems; ++r) {
      const int64_t p = base + r * kThreads + threadIdx.x;
      if (p < end) atomicAdd(&h[lv.digit(k[r])], 1u);
    }
    __syncthreads();
    uint32_t* out = lv.hist + (int64_t(it.hist0) + tt) * 256;
    for (int d = threadIdx.x; d < 256; d += kThreads) out[d] = h[d];
    __syncthreads();
  }
}

// Exclusive scan over the (digit, tile) counts of one item, digit-major (a
// thread per digit walks the tiles, whose rows of 256 counts it reads
// together with its neighbours), then the item's buckets become chunks (at
// most kSortLocalMax entries, packed greedily in digit order) or items of
// the next level.  The greedy packing is a chain of "next chunk starts at
// digit e" steps: every thread finds its e by a binary search in the bucket
// starts, one thread follows the chain (one step per chunk), and all write
// the chunks.  (One thread walking the 256 digits twice took 8 us of a
// block: 15.5 ms of a wide index's 118 ms of sorting.)
__global__ void __launch_bounds__(256) k_sort_scan(Level lv) {
  __shared__ uint32_t pre[257];              // bucket starts, relative to the item
  __shared__ uint32_t wsum[8], bigm[8];      // per warp: total, mask of large buckets
  __shared__ uint16_t nxt[256];
  __shared__ uint8_t head[256];              // a chunk or item starts at this digit
  __shared__ uint32_t chunk0;
  const uint32_t ni = min(lv.cnt[2 * lv.t], lv.item_cap);
  const int d = threadIdx.x, lane = d & 31, warp = d >> 5;
  const bool last_level = lv.t + 1 >= lv.K;
  for (uint32_t item = blockIdx.x; item < ni; item += gridDim.x) {
    const SortItem it = lv.items[item];
    const uint32_t tiles = ntiles(it.size);
    if (it.seg >= uint32_t(lv.segs) || int64_t(it.start) + it.size > lv.M ||
        int64_t(it.hist0) + tiles > int64_t(lv.tile_cap))
      continue;                                   // only after an overflow
    uint32_t* hs = lv.hist + int64_t(it.hist0) * 256 + d;
    uint32_t s = 0, t0 = 0;
    for (; t0 + 8 <= tiles; t0 += 8) {          // eight independent loads in flight
      uint32_t c[8];
#pragma unroll
      for (int q = 0; q < 8; ++q) c[q] = hs[(t0 + q) * 256];
#pragma unroll
      for (int q = 0; q < 8; ++q) s += c[q];
    }
    for (; t0 < tiles; ++t0) s += hs[t0 * 256];
    // exclusive scan of the 256 digit totals
    uint32_t incl = s;
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t u = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl += u;
    }
    const bool big = s > uint32_t(kSortLocalMax);
    const uint32_t bm = __ballot_sync(0xffffffffu, big);
    if (lane == 31) {
      wsum[warp] = incl;
      bigm[warp] = bm;
    }
    head[d] = 0;
    __syncthreads();
    uint32_t before = 0;
#pragma unroll
    for (int q = 0; q < 8; ++q) before += q < warp ? wsum[q] : 0u;
    const uint32_t start = before + incl - s;
    pre[d] = start;
    if (d == 255) pre[256] = start + s;
    uint32_t run = start;
    t0 = 0;
    for (; t0 + 8 <= tiles; t0 += 8) {
      uint32_t c[8];
#pragma unroll
      for (int q = 0; q < 8; ++q) c[q] = hs[(t0 + q) * 256];
#pragma unroll
      for (int q = 0; q < 8; ++q) {
        hs[(t0 + q) * 256] = run;
        run += c[q];
      }
    }
    for (; t0 < tiles; ++t0) {
      const uint32_t c = hs[t0 * 256];
      hs[t0 * 256] = run;
      run += c;
    }
    __syncthreads();
    // where the chunk that starts at digit d ends: before the next large
    // bucket, and while at most kSortLocalMax entries are in it
    int e = d + 1;
    if (!big) {
      int stop = 256;
      for (int q = 7; q >= warp; --q) {
        const uint32_t m = q == warp ? bigm[q] & ~((1u << lane) - 1u) : bigm[q];
        if (m) stop = q * 32 + __ffs(m) - 1;
      }
      int hi = stop;
      while (e < hi) {
        const int mid = (e + hi + 1) >> 1;
        if (pre[mid] - start <= uint32_t(kSortLocalMax)) e = mid;
        else hi = mid - 1;
      }
    }
    nxt[d] = uint16_t(e);
    __syncthreads();
    if (d == 0)
      for (int g = 0; g < 256; g = nxt[g]) head[g] = 1;
    __syncthreads();
    const uint32_t size = pre[e] - start;
    const bool lead = head[d] != 0 && size > 0;
    const bool is_item = lead && big && !last_level;
    const bool is_chunk = lead && !is_item;
    // a bucket's first entry shares t hash values with its predecessor (the
    // item's own first entry keeps the item's count)
    const uint32_t l0 = start == 0 ? it.lcp0 : uint32_t(lv.t);
    const uint32_t cm = __ballot_sync(0xffffffffu, is_chunk);
    if (lane == 0) wsum[warp] = __popc(cm);
    __syncthreads();
    if (d == 0) {
      uint32_t n = 0;
      for (int q = 0; q < 8; ++q) n += wsum[q];
      chunk0 = n ? atomicAdd(&lv.cnt[kCntChunks], n) : 0u;
    }
    __syncthreads();
    if (is_chunk) {
      uint32_t slot = chunk0 + __popc(cm & ((1u << lane) - 1u));
      for (int q = 0; q < warp; ++q) slot += wsum[q];
      if (slot < lv.chunk_cap) {
        SortChunk ch;
        ch.seg = it.seg;
        ch.start = it.start + start;
        ch.size = size;
        ch.lcp0 = uint8_t(l0);
        ch.buf = uint8_t(lv.t & 1);
        ch.equal = uint8_t(big);                // after the last level: equal keys, already in order
        ch.t = uint8_t(lv.t);
        lv.chunks[slot] = ch;
      } else {
        lv.cnt[kCntOverflow] = 1u;
      }
    }
    if (is_item) {
      const uint32_t nt = ntiles(size);
      const uint32_t slot = atomicAdd(&lv.cnt[2 * (lv.t + 1)], 1u);
      const uint32_t tb = atomicAdd(&lv.cnt[2 * (lv.t + 1) + 1], nt);
      if (slot < lv.item_cap && tb + nt <= lv.tile_cap) {
        lv.items_next[slot] = SortItem{it.seg, it.start + start, size, tb, l0, {0u, 0u, 0u}};
        for (uint32_t q = 0; q < nt; ++q) lv.tile_next[tb + q] = (uint64_t(q) << 32) | slot;
      } else {
        lv.cnt[kCntOverflow] = 1u;
      }
    }
    __syncthreads();
  }
}

__global__ void __launch_bounds__(kThreads) k_sort_scatter(Level lv) {
  __shared__ uint32_t wh[kWarps][256];
  __shared__ uint32_t loff[256];             // tile-local start of each digit
  __shared__ uint64_t sk[kTile];             // the tile in digit order
  __shared__ uint32_t sv[kTile];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const uint32_t lt = (1u << lane) - 1u;
  const uint32_t nt = min(lv.cnt[2 * lv.t + 1], lv.tile_cap);
  for (uint32_t tile = blockIdx.x; tile < nt; tile += gridDim.x) {
    SortItem it;
    uint32_t tt;
    if (!lv.tile_of(tile, it, tt)) continue;
    for (int q = threadIdx.x; q < kWarps * 256; q += kThreads) (&wh[0][0])[q] = 0;
    __syncthreads();
    const int64_t end = int64_t(it.start) + it.size;
    const int64_t base = int64_t(it.start) + int64_t(tt) * kTile + int64_t(warp) * kWarpSpan;
    uint64_t key[kRounds];
    uint32_t val[kRounds], dig[kRounds], loc[kRounds];
    // all loads of the warp's span first (independent, in flight together)
#pragma unroll
    for (int r = 0; r < kRounds; ++r) {
      const int64_t p = base + r * 32 + lane;
      key[r] = 0;
      val[r] = 0;
      if (p < end) lv.load(it.seg, p, key[r], val[r]);
    }
#pragma unroll
    for (int r = 0; r < kRounds; ++r) {
      const int64_t p = base + r * 32 + lane;
      // out of range: a digit no valid entry has
      const uint32_t dg = p < end ? lv.digit(key[r]) : 256u + lane;
      dig[r] = dg;
      const uint32_t peers = __match_any_sync(0xffffffffu, dg);
      const uint32_t rank = __popc(peers & lt);
      const uint32_t cnt = __popc(peers);
      uint32_t b = 0;
      if (dg < 256u) b = wh[warp][dg];
      __syncwarp();
      if (dg < 256u && rank == 0) wh[warp][dg] = b + cnt;
      __syncwarp();
      loc[r] = b + rank;
    }
    __syncthreads();
    for (int d = threadIdx.x; d < 256; d += kThreads) {
      uint32_t run = 0;
      for (int w = 0; w < kWarps; ++w) {
        const uint32_t c = wh[w][d];
        wh[w][d] = run;
        run += c;
      }
      loff[d] = run;                           // digit total, scanned below
    }
    __syncthreads();
    if (threadIdx.x < 32) {                    // exclusive scan of the 256 totals
      uint32_t v[8], run = 0;
#pragma unroll
      for (int q = 0; q < 8; ++q) { v[q] = loff[lane * 8 + q]; run += v[q]; }
      uint32_t incl = run;
      for (int o = 1; o < 32; o <<= 1) {
        const uint32_t u = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += u;
      }
      uint32_t b = incl - run;
#pragma unroll
      for (int q = 0; q < 8; ++q) { loff[lane * 8 + q] = b; b += v[q]; }
    }
    __syncthreads();
    // the tile in digit order in shared memory (stable within each digit) ...
#pragma unroll
    for (int r = 0; r < kRounds; ++r) {
      if (dig[r] < 256u) {
        const uint32_t q = loff[dig[r]] + wh[warp][dig[r]] + loc[r];
        sk[q] = key[r];
        sv[q] = val[r];
      }
    }
    __syncthreads();
    // ... then written out in that order: runs of equal digits are contiguous
    const uint32_t* hs = lv.hist + (int64_t(it.hist0) + tt) * 256;
    const int64_t n_tile = min(int64_t(kTile), end - (int64_t(it.start) + int64_t(tt) * kTile));
    const int64_t obase = int64_t(it.seg) * lv.M + it.start;
    for (int q = threadIdx.x; q < n_tile; q += kThreads) {
      const uint64_t k = sk[q];
      const uint32_t d = lv.digit(k);
      const uint32_t dst = hs[d] + (uint32_t(q) - loff[d]);
      lv.kout[obase + dst] = k;
      lv.vout[obase + dst] = sv[q];
    }
    __syncthreads();
  }
}

struct LocalArgs {
  const uint64_t* k[2];
  const uint32_t* v[2];
  const SortChunk* chunks;
  uint32_t* cnt;
  uint32_t chunk_cap;
  int64_t M;
  int D, j0, K, segs;
  uint64_t kmask;                 // the K leading bytes of a key
  uint32_t* order;
  uint8_t* lcp;
};

// Each chunk sorted completely in shared memory by (key, window), then
// order and common-prefix lengths written to their final ranks.
//
// The entries are first spread over 2048 bins, about one per entry, by the
// first three hash values that differ inside the chunk, each as its offset
// from the chunk's smallest there in the bits its range needs, most
// significant first (monotone in the key).  Then every entry
// counts the smaller ones in its bin.  (key, window) is a total order, so
// neither step has to be stable: one shared-memory atomic per entry, no
// match masks.  On the hash strings of z-normalised windows an entry's bin
// holds 6 to 7 entries (mean over entries).  Chunks whose bins are crowded
// (sum of squared sizes above 48 per entry: equal or nearly equal keys) are
// sorted by a bitonic network instead; chunks whose keys differ in no value
// below the partitioned one are in order already.
//
// The least-significant-digit form before (6 to 7 digit passes with match
// masks over 8-bit digits) took 9.0 ms for 1.6e8 entries, this one 3.0; it
// is bound by issue (the compares inside the bins come first).
__global__ void __launch_bounds__(kLocalThreads, kLocalBlocks) k_sort_local(LocalArgs a) {
  __shared__ uint64_t sk[kSortLocalMax];
  __shared__ uint32_t sv[kSortLocalMax];
  __shared__ uint32_t bin0[kBins + 1];       // counts, then first ranks
  __shared__ uint16_t sb[kSortLocalMax];     // bin of the entry
  __shared__ uint32_t s_diff[2], s_min[3], s_max[3], s_cnt[kLocalWarps], s_sq[kLocalWarps];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const uint32_t nc = min(a.cnt[kCntChunks], a.chunk_cap);
  for (uint32_t c = blockIdx.x; c < nc; c += gridDim.x) {
    const SortChunk ch = a.chunks[c];
    if (ch.seg >= uint32_t(a.segs) || int64_t(ch.start) + ch.size > a.M) continue;   // only after an overflow
    const int64_t ib = int64_t(ch.seg) * a.M + ch.start;
    const int64_t ob = (int64_t(a.j0) * a.D + ch.seg) * a.M + ch.start;
    const uint64_t* kin = (ch.buf ? a.k[1] : a.k[0]) + ib;
    const uint32_t* vin = (ch.buf ? a.v[1] : a.v[0]) + ib;
    const int n = int(ch.size);
    if (ch.equal || n > kSortLocalMax) {
      // equal keys (after the last level): already in order
      for (int q = tid; q < n; q += kLocalThreads) {
        a.order[ob + q] = vin[q];
        a.lcp[ob + q] = q == 0 ? ch.lcp0 : uint8_t(a.K);
      }
      continue;
    }
    uint64_t k[kLocalItems];
    uint32_t v[kLocalItems];
    if (tid < 2) s_diff[tid] = 0u;
    if (tid < 3) {
      s_min[tid] = ~0u;
      s_max[tid] = 0u;
    }
    // the bits in which any two keys differ
    const uint64_t k0 = kin[0] & a.kmask;
    uint64_t diff = 0;
#pragma unroll
    for (int i = 0; i < kLocalItems; ++i) {
      const int q = i * kLocalThreads + tid;
      k[i] = q < n ? kin[q] & a.kmask : ~0ull;
      v[i] = q < n ? vin[q] : ~0u;
      diff |= q < n ? k[i] ^ k0 : 0ull;
    }
#pragma unroll
    for (int q = 0; q < kBins / kLocalThreads; ++q) bin0[q * kLocalThreads + tid] = 0u;
    const uint32_t d0 = __reduce_or_sync(0xffffffffu, uint32_t(diff >> 32));
    const uint32_t d1 = __reduce_or_sync(0xffffffffu, uint32_t(diff));
    __syncthreads();
    if (lane == 0) {
      atomicOr(&s_diff[0], d0);
      atomicOr(&s_diff[1], d1);
    }
    __syncthreads();
    diff = (uint64_t(s_diff[0]) << 32) | s_diff[1];
    // no value below the partitioned one differs: in order as it is
    const bool sorted = ch.t >= 7 || (diff & (~0ull >> (8 * (int(ch.t) + 1)))) == 0ull;
    // the first three hash values that differ (as shifts), their ranges
    int sh[3];
    {
      uint64_t rest = diff;
#pragma unroll
      for (int f = 0; f < 3; ++f) {
        sh[f] = rest ? (63 - __clzll(static_cast<long long>(rest))) & ~7 : 0;
        rest &= (1ull << sh[f]) - 1ull;
      }
    }
    uint32_t lo[3] = {~0u, ~0u, ~0u}, hi[3] = {0u, 0u, 0u};
#pragma unroll
    for (int i = 0; i < kLocalItems; ++i)
      if (i * kLocalThreads + tid < n) {
#pragma unroll
        for (int f = 0; f < 3; ++f) {
          const uint32_t x = uint32_t(k[i] >> sh[f]) & 255u;
          lo[f] = min(lo[f], x);
          hi[f] = max(hi[f], x);
        }
      }
#pragma unroll
    for (int f = 0; f < 3; ++f) {
      lo[f] = __reduce_min_sync(0xffffffffu, lo[f]);
      hi[f] = __reduce_max_sync(0xffffffffu, hi[f]);
      if (lane == 0) {
        atomicMin(&s_min[f], lo[f]);
        atomicMax(&s_max[f], hi[f]);
      }
    }
    __syncthreads();
    // bin: ((x0 - lo0) in w0 bits, (x1 - lo1) in w1, (x2 - lo2) in w2), its
    // leading kBinBits bits.  A shift of 0 is a value taken already, or a
    // position all keys share: no bits
    int up[3], bits = 0;
#pragma unroll
    for (int f = 2; f >= 0; --f) {
      lo[f] = s_min[f];
      const bool use = f == 0 ? diff != 0 : sh[f] < sh[f - 1];
      up[f] = use ? bits : 32;
      if (use) bits += 32 - __clz(int(s_max[f] - lo[f]));
    }
    const int drop = bits > kBinBits ? bits - kBinBits : 0;
    auto bin_of = [&](uint64_t key) {
      uint32_t z = 0;
#pragma unroll
      for (int f = 0; f < 3; ++f)
        if (up[f] < 32) z |= ((uint32_t(key >> sh[f]) & 255u) - lo[f]) << up[f];
      return z >> drop;
    };
    bool spread = false;
    if (!sorted) {
      uint32_t br[kLocalItems];              // bin << 16 | rank of arrival
#pragma unroll
      for (int i = 0; i < kLocalItems; ++i) {
        br[i] = 0;
        if (i * kLocalThreads + tid < n) {
          const uint32_t b = bin_of(k[i]);
          br[i] = (b << 16) | atomicAdd(&bin0[b], 1u);
        }
      }
      __syncthreads();
      // first ranks of the bins, and the sum of their squared sizes
      uint32_t cnt[kBins / kLocalThreads], run = 0, sq = 0;
#pragma unroll
      for (int q = 0; q < kBins / kLocalThreads; ++q) {
        cnt[q] = bin0[tid * (kBins / kLocalThreads) + q];
        run += cnt[q];
        sq += cnt[q] * cnt[q];
      }
      uint32_t incl = run;
      for (int o = 1; o < 32; o <<= 1) {
        const uint32_t u = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += u;
      }
      sq = __reduce_add_sync(0xffffffffu, sq);
      if (lane == 31) {
        s_cnt[warp] = incl;
        s_sq[warp] = sq;
      }
      __syncthreads();
      uint32_t first = incl - run, all_sq = 0;
#pragma unroll
      for (int w = 0; w < kLocalWarps; ++w) {
        if (w < warp) first += s_cnt[w];
        all_sq += s_sq[w];
      }
#pragma unroll
      for (int q = 0; q < kBins / kLocalThreads; ++q) {
        bin0[tid * (kBins / kLocalThreads) + q] = first;
        first += cnt[q];
      }
      if (tid == kLocalThreads - 1) bin0[kBins] = first;
      spread = all_sq <= 48u * uint32_t(n);
      __syncthreads();
      if (spread) {
#pragma unroll
        for (int i = 0; i < kLocalItems; ++i)
          if (i * kLocalThreads + tid < n) {
            const uint32_t p = bin0[br[i] >> 16] + (br[i] & 0xffffu);
            sk[p] = k[i];
            sv[p] = v[i];
            sb[p] = uint16_t(br[i] >> 16);
          }
        __syncthreads();
        // ranks inside the bins (neighbouring threads read the same bins)
        uint32_t to[kLocalItems];
#pragma unroll
        for (int i = 0; i < kLocalItems; ++i) {
          const int p = i * kLocalThreads + tid;
          if (p >= n) continue;
          k[i] = sk[p];
          v[i] = sv[p];
          const uint32_t b = sb[p];
          const uint32_t q0 = bin0[b], q1 = bin0[b + 1];
          uint32_t r = q0;
          for (uint32_t q = q0; q < q1; ++q) {
            const uint64_t o = sk[q];
            r += o < k[i] ? 1u : 0u;
            if (o == k[i] && q != uint32_t(p)) r += sv[q] < v[i] ? 1u : 0u;
          }
          to[i] = r;
        }
        __syncthreads();
#pragma unroll
        for (int i = 0; i < kLocalItems; ++i)
          if (i * kLocalThreads + tid < n) {
            sk[to[i]] = k[i];
            sv[to[i]] = v[i];
          }
      }
    }
    if (!spread) {
      // as loaded; the places past n hold the largest (key, window)
#pragma unroll
      for (int i = 0; i < kLocalItems; ++i) {
        sk[i * kLocalThreads + tid] = k[i];
        sv[i * kLocalThreads + tid] = v[i];
      }
      if (!sorted) {
        int m = 2;
        while (m < n) m <<= 1;
        for (int len = 2; len <= m; len <<= 1)
          for (int st = len >> 1; st > 0; st >>= 1) {
            __syncthreads();
            for (int q = tid; q < m / 2; q += kLocalThreads) {
              const int x = 2 * st * (q / st) + q % st, y = x + st;
              const uint64_t kx = sk[x], ky = sk[y];
              const uint32_t vx = sv[x], vy = sv[y];
              const bool gt = kx > ky || (kx == ky && vx > vy);
              if (gt == ((x & len) == 0)) {
                sk[x] = ky; sk[y] = kx;
                sv[x] = vy; sv[y] = vx;
              }
            }
          }
      }
    }
    __syncthreads();
    for (int q = tid; q < n; q += kLocalThreads) {
      a.order[ob + q] = sv[q];
      uint32_t l = ch.lcp0;
      if (q > 0) l = min(uint32_t(__clzll(static_cast<long long>(sk[q] ^ sk[q - 1]))) >> 3, uint32_t(a.K));
      a.lcp[ob + q] = uint8_t(l);
    }
    __syncthreads();
  }
}

}  // namespace

SortScratch sort_scratch_carve(void* base, int64_t M, int segs) {
  const SortCaps c = sort_caps(M, segs);
  const int64_t e = M * segs;
  const auto up = sort_up256;
  unsigned char* p = static_cast<unsigned char*>(base);
  SortScratch sc;
  sc.k0 = reinterpret_cast<uint64_t*>(p); p += up(size_t(e) * 8);
  sc.k1 = reinterpret_cast<uint64_t*>(p); p += up(size_t(e) * 8);
  sc.v0 = reinterpret_cast<uint32_t*>(p); p += up(size_t(e) * 4);
  sc.v1 = reinterpret_cast<uint32_t*>(p); p += up(size_t(e) * 4);
  sc.hist = reinterpret_cast<uint32_t*>(p); p += up(size_t(c.tile_cap) * 256 * 4);
  sc.items[0] = reinterpret_cast<SortItem*>(p); p += up(size_t(c.item_cap) * sizeof(SortItem));
  sc.items[1] = reinterpret_cast<SortItem*>(p); p += up(size_t(c.item_cap) * sizeof(SortItem));
  sc.tile_item[0] = reinterpret_cast<uint64_t*>(p); p += up(size_t(c.tile_cap) * 8);
  sc.tile_item[1] = reinterpret_cast<uint64_t*>(p); p += up(size_t(c.tile_cap) * 8);
  sc.chunks = reinterpret_cast<SortChunk*>(p); p += up(size_t(c.chunk_cap) * sizeof(SortChunk));
  sc.cnt = reinterpret_cast<uint32_t*>(p);
  sc.cap_entries = e;
  sc.caps = c;
  sc.M = M;
  sc.segs = segs;
  return sc;
}

cudaError_t launch_sort_reps(const Index& ix, int j0, int j1, const SortScratch& sc,
                             cudaStream_t s) {
  if (j1 <= j0) return cudaSuccess;
  const int segs = (j1 - j0) * ix.D;
  if (sc.M != ix.M || segs > sc.segs) return cudaErrorInvalidValue;
  const SortCaps& c = sc.caps;
  cudaError_t e = cudaSuccess;
  const int64_t tpm = (ix.M + kTile - 1) / kTile;
  const int sm = sm_count();
  {
    const int64_t total = int64_t(segs) * tpm;
    const int g = int(std::min<int64_t>((total + 255) / 256, int64_t(sm) * 8));
    MOMENTI_LAUNCH("sort_init", s, k_sort_init<<<std::max(g, 1), 256, 0, s>>>(segs, ix.M, sc.items[0], sc.tile_item[0], sc.cnt));
  }
  uint32_t n_items = uint32_t(segs), n_tiles = uint32_t(int64_t(segs) * tpm);
  const bool host = sc.host_cnt != nullptr;
  for (int t = 0; t < ix.K; ++t) {
    Level lv;
    lv.keys = ix.keys;
    lv.kin = t ? (((t - 1) & 1) ? sc.k1 : sc.k0) : nullptr;
    lv.vin = t ? (((t - 1) & 1) ? sc.v1 : sc.v0) : nullptr;
    lv.kout = (t & 1) ? sc.k1 : sc.k0;
    lv.vout = (t & 1) ? sc.v1 : sc.v0;
    lv.M = ix.M;
    lv.D = ix.D;
    lv.j0 = j0;
    lv.t = t;
    lv.K = ix.K;
    lv.segs = segs;
    lv.items = sc.items[t & 1];
    lv.items_next = sc.items[(t + 1) & 1];
    lv.tile_item = sc.tile_item[t & 1];
    lv.tile_next = sc.tile_item[(t + 1) & 1];
    lv.hist = sc.hist;
    lv.chunks = sc.chunks;
    lv.cnt = sc.cnt;
    lv.item_cap = uint32_t(c.item_cap);
    lv.tile_cap = uint32_t(c.tile_cap);
    lv.chunk_cap = uint32_t(c.chunk_cap);
    // with the host in the loop the grids are exact; without it, the
    // largest a level can need (the kernels stop at the device counts)
    const unsigned gt = unsigned(std::max<int64_t>(1, host ? n_tiles : c.tile_cap));
    const unsigned gi = unsigned(std::max<int64_t>(1, host ? n_items : c.item_cap));
    MOMENTI_LAUNCH("sort_hist", s, k_sort_hist<<<gt, kThreads, 0, s>>>(lv));
    MOMENTI_LAUNCH("sort_scan", s, k_sort_scan<<<gi, 256, 0, s>>>(lv));
    MOMENTI_LAUNCH("sort_scatter", s, k_sort_scatter<<<gt, kThreads, 0, s>>>(lv));
    if (host) {
      e = cudaMemcpyAsync(sc.host_cnt, sc.cnt, 32 * sizeof(uint32_t), cudaMemcpyDeviceToHost, s);
      if (e != cudaSuccess) return e;
      e = cudaStreamSynchronize(s);
      if (e != cudaSuccess) return e;
      if (sc.host_cnt[kCntOverflow]) return cudaErrorInvalidValue;   // capacities are bounds: not expected
      n_items = sc.host_cnt[2 * (t + 1)];
      n_tiles = sc.host_cnt[2 * (t + 1) + 1];
      if (n_items == 0) break;
    }
  }
  LocalArgs la;
  la.k[0] = sc.k0;
  la.k[1] = sc.k1;
  la.v[0] = sc.v0;
  la.v[1] = sc.v1;
  la.chunks = sc.chunks;
  la.cnt = sc.cnt;
  la.chunk_cap = uint32_t(c.chunk_cap);
  la.M = ix.M;
  la.D = ix.D;
  la.j0 = j0;
  la.K = ix.K;
  la.segs = segs;
  la.kmask = ix.K >= 8 ? ~0ull : ~((~0ull) >> (8 * ix.K));
  la.order = ix.order;
  la.lcp = ix.lcp;
  // four CTAs of 8 warps per SM (register bound; five spill); chunks
  // statically interleaved over them
  MOMENTI_LAUNCH("sort_local", s, k_sort_local<<<sm * kLocalBlocks, kLocalThreads, 0, s>>>(la));
  return cudaGetLastError();
}

}  // namespace momenti

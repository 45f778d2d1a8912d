// Row-level utilities outside the super step: relabelling a CSR into another
// row order and node numbering (with each row sorted), input validation and
// the canonical edge export (Section 2: ordered
// edges [a,b], a<b).
#include <algorithm>

#include "cb_internal.cuh"
#include "pair_lists.cuh"
#include "team.cuh"

namespace cb {
namespace {

constexpr int kRowWarpMax = 256;     // rows up to this length: one warp
constexpr int kRowBlockSmem = 16384; // rows up to this length: one CTA in shared memory

__device__ __forceinline__ void latch(int32_t* err, int32_t code) { atomicCAS(err, 0, code); }

// A warp on up to 32 consecutive rows r0.. as one run of entries: every lane owns a row's offset, lanes take consecutive entries
// whatever their rows, and kTileLoads loads are in flight per lane.  A warp per
// row instead waits for two offsets, then for the entries, with most lanes
// idle on rows of 10 to 100 entries.
constexpr int kTileLoads = 4;
struct RowTile {
  int64_t r0, off, end;   // first row; this lane's row offset; the tile's end
  int lane;
  __device__ __forceinline__ RowTile(const int64_t* __restrict__ rp, int64_t n, int64_t first, int rows = 32)
      : r0(first), lane(threadIdx.x & 31) {
    const int64_t last = first + rows < n ? first + rows : n;
    off = rp[first + lane < last ? first + lane : last];
    end = rp[last];
  }
  __device__ __forceinline__ int64_t begin() const { return __shfl_sync(kFull, off, 0); }
  // the row (relative to r0) of entry e >= begin(): the last one whose offset is <= e
  __device__ __forceinline__ int row_of(int64_t e) const {
    int k = 0;
#pragma unroll
    for (int s = 16; s; s >>= 1) {
      const int64_t o = __shfl_sync(kFull, off, k + s);
      if (o <= e) k += s;
    }
    return k;
  }
};

// Where a tile's runs are independent, tile_split warps share a tile, each
// taking every such run, so that on small graphs a tile with a hub does not
// keep one warp busy alone (relabelling n=2^17: 55 -> 40 us; at n=2^25, with
// tiles enough, 18.7 -> 23.3 ms, so not there).
int tile_split(int per) { return per < 32 ? 4 : 1; }

// Rows per warp: 32, fewer where that would leave
// warps without rows (n=4096: 32 rows per warp took 85 us for the export, 4 rows 60).
int rows_per_warp(int64_t n, int num_sms) {
  int64_t r = 32;
  while (r > 4 && (n + r - 1) / r < int64_t(num_sms) * 64) r >>= 1;
  return static_cast<int>(r);
}

struct RowArgs {
  int64_t nrows;
  const int64_t* src_rp;
  const int32_t* src_col;
  const int32_t* rowmap;
  const int32_t* valmap;
  const int64_t* dst_rp;
  int32_t* dst_col;
  int32_t* err;
};

template <class Team>
__device__ void relabel_row(Team& tm, const RowArgs& a, int64_t q, int32_t* buf) {
  const int64_t x = a.rowmap ? a.rowmap[q] : q;
  const int64_t s0 = a.src_rp[x], len = a.src_rp[x + 1] - s0;
  const int64_t d0 = a.dst_rp[q];
  if (len != a.dst_rp[q + 1] - d0) {
    if (tm.rank == 0) latch(a.err, kErrRowLength);
    return;
  }
  const int P = next_pow2(static_cast<int>(len));
  for (int i = tm.rank; i < P; i += Team::N) {
    int32_t v = 0x7fffffff;
    if (i < len) {
      v = a.src_col[s0 + i];
      if (a.valmap) v = a.valmap[v];
    }
    buf[i] = v;
  }
  tm.sync();
  team_bitonic_sort(tm, buf, P);
  for (int i = tm.rank; i < len; i += Team::N) a.dst_col[d0 + i] = buf[i];
  tm.sync();
}

__global__ void __launch_bounds__(256) k_rows_warp(RowArgs a) {
  __shared__ int32_t buf[8][kRowWarpMax];
  WarpTeam tm;
  const int w = threadIdx.x >> 5;
  const int64_t nw = int64_t(gridDim.x) * 8;
  for (int64_t q = blockIdx.x * int64_t(8) + w; q < a.nrows; q += nw) {
    const int64_t len = a.dst_rp[q + 1] - a.dst_rp[q];
    if (len > kRowWarpMax) continue;
    relabel_row(tm, a, q, buf[w]);
  }
}

// Long rows: one CTA per row, shared memory or a global slice per CTA.
__global__ void __launch_bounds__(256) k_rows_block(RowArgs a, int32_t* gws, int64_t slice) {
  extern __shared__ int32_t sbuf[];
  __shared__ int64_t red[BlockTeam<256>::kRedSlots];
  BlockTeam<256> tm(red);
  for (int64_t q = blockIdx.x; q < a.nrows; q += gridDim.x) {
    const int64_t len = a.dst_rp[q + 1] - a.dst_rp[q];
    if (len <= kRowWarpMax) continue;
    int32_t* buf = (len <= kRowBlockSmem) ? sbuf : gws + slice * blockIdx.x;
    relabel_row(tm, a, q, buf);
  }
}

// Validation of the input: rows strictly increasing, in range, no self loop,
// and symmetric.  Symmetry is checked exactly:
//   - the entries above the diagonal, summed over all rows, are as many as
//     those below;
//   - every entry y > x of row x is found among the entries of row y below
//     the diagonal (L_y).
// The found entries are distinct (rows are strictly increasing), so each L_y
// holds at least as many as point into it, and the totals force equality.
// Small graphs are checked in place; for larger ones the upper entries
// are first partitioned into buckets of target rows, so that each bucket's
// searches stay within a few MB of rows.

constexpr int kVBuckets = 4096;     // target-row buckets of the partition

// The partition: CTA c takes a range of tiles, counts its upper entries per
// bucket (k_scan_rows), and, after a scan over (bucket, CTA), writes them there
// (k_vpart): the entries are read twice in all.
constexpr int kVThreads = 512;

// A tile's kept lanes (a ballot at run eb..eb+31) that belong to this lane's row.
__device__ __forceinline__ int own_count(const RowTile& tile, int64_t eb, unsigned kept) {
  const int64_t nx = __shfl_down_sync(kFull, tile.off, 1);
  const int64_t lo = tile.off - eb, hi = (tile.lane == 31 ? tile.end : nx) - eb;
  if (hi <= 0 || lo >= 32) return 0;
  const unsigned from = lo > 0 ? ~((1u << lo) - 1u) : ~0u;
  const unsigned to = hi < 32 ? (1u << hi) - 1u : ~0u;
  return __popc(kept & from & to);
}

// What the first pass over the rows finds, in the handle's scratch words.
enum { kScanMaxdeg = 0, kScanUnsorted, kScanBad, kScanUpper, kScanLower, kScanWords };

// The first pass over the entries: ids, order, entries on each side of the
// diagonal, low[x] = those of row x below it (its first entries when the row
// is sorted), and, for the partition (kHist), the upper entries per bucket and
// CTA.  Does nothing when the offsets were bad.
template <bool kHist>
__global__ void __launch_bounds__(kVThreads) k_scan_rows(int64_t n, const int64_t* __restrict__ rp,
                                                         const int32_t* __restrict__ col, int per, int sh, int nb,
                                                         int32_t* __restrict__ counts, int32_t* __restrict__ low,
                                                         unsigned long long* __restrict__ found, const int32_t* err) {
  __shared__ int32_t cnt[kHist ? kVBuckets : 1];
  __shared__ unsigned long long sums[2];
  if (*err != 0) return;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  // CTA ranges of tiles for the partition, else tiles spread over the CTAs
  const int64_t tiles = (n + per - 1) / per, each = (tiles + gridDim.x - 1) / gridDim.x;
  const int64_t t0 = kHist ? blockIdx.x * each : blockIdx.x, step = kHist ? 1 : gridDim.x;
  const int64_t t1 = kHist && t0 + each < tiles ? t0 + each : tiles;
  if (kHist)
    for (int b = threadIdx.x; b < nb; b += blockDim.x) cnt[b] = 0;
  if (threadIdx.x < 2) sums[threadIdx.x] = 0;
  __syncthreads();
  bool unsorted = false, bad = false;
  unsigned long long up = 0, down = 0;
  for (int64_t t = t0 + w * step; t < t1; t += step * (kVThreads / 32)) {
    const RowTile tile(rp, n, per * t, per);
    int c = 0;
    for (int64_t e0 = tile.begin(); e0 < tile.end; e0 += 32 * kTileLoads) {
      int32_t y[kTileLoads], before[kTileLoads];
#pragma unroll
      for (int j = 0; j < kTileLoads; ++j) {
        const int64_t e = e0 + 32 * j + lane;
        y[j] = e < tile.end ? col[e] : 0;
        before[j] = e < tile.end && lane == 0 && e > 0 ? col[e - 1] : 0;
      }
#pragma unroll
      for (int j = 0; j < kTileLoads; ++j) {
        const int64_t e = e0 + 32 * j + lane;
        const int k = tile.row_of(e);
        const int64_t first = __shfl_sync(kFull, tile.off, k);
        int32_t prev = __shfl_up_sync(kFull, y[j], 1);
        if (lane == 0) prev = before[j];
        const bool in = e < tile.end;
        const int64_t x = tile.r0 + k;
        const bool wrong = y[j] < 0 || y[j] >= n || y[j] == x;
        bad |= in && wrong;
        unsorted |= in && e > first && prev >= y[j];
        const bool above = in && !wrong && y[j] > x;
        const unsigned lower = __ballot_sync(kFull, in && !wrong && y[j] < x);
        c += own_count(tile, e0 + 32 * j, lower);
        up += above;
        if (kHist && above) atomicAdd(&cnt[y[j] >> sh], 1);
      }
    }
    if (lane < per && tile.r0 + lane < n) {
      low[tile.r0 + lane] = c;
      down += c;
    }
  }
  if (__any_sync(kFull, unsorted) && lane == 0) found[kScanUnsorted] = 1;
  if (__any_sync(kFull, bad) && lane == 0) found[kScanBad] = 1;
#pragma unroll
  for (int o = 16; o; o >>= 1) {
    up += __shfl_xor_sync(kFull, up, o);
    down += __shfl_xor_sync(kFull, down, o);
  }
  if (lane == 0) {
    atomicAdd(&sums[0], up);
    atomicAdd(&sums[1], down);
  }
  __syncthreads();
  if (threadIdx.x < 2 && sums[threadIdx.x]) atomicAdd(found + kScanUpper + threadIdx.x, sums[threadIdx.x]);
  if (kHist)
    for (int b = threadIdx.x; b < nb; b += blockDim.x) counts[int64_t(b) * gridDim.x + blockIdx.x] = cnt[b];
}

// The upper entries (x, y) into their places; slots past `cap` (more upper
// entries than a symmetric graph has) latch the error.
__global__ void __launch_bounds__(kVThreads) k_vpart(int64_t n, const int64_t* __restrict__ rp,
                                                     const int32_t* __restrict__ col, int sh, int nb,
                                                     const int64_t* __restrict__ place, int2* __restrict__ part,
                                                     int64_t cap, int32_t* err) {
  __shared__ unsigned long long cur[kVBuckets];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int64_t tiles = (n + 31) / 32, per = (tiles + gridDim.x - 1) / gridDim.x;
  const int64_t t0 = blockIdx.x * per, t1 = t0 + per < tiles ? t0 + per : tiles;
  for (int b = threadIdx.x; b < nb; b += blockDim.x)
    cur[b] = static_cast<unsigned long long>(place[int64_t(b) * gridDim.x + blockIdx.x]);
  __syncthreads();
  for (int64_t t = t0 + w; t < t1; t += kVThreads / 32) {
    const RowTile tile(rp, n, 32 * t);
    for (int64_t e0 = tile.begin(); e0 < tile.end; e0 += 32 * kTileLoads) {
      int32_t y[kTileLoads];
#pragma unroll
      for (int j = 0; j < kTileLoads; ++j) {
        const int64_t e = e0 + 32 * j + lane;
        y[j] = e < tile.end ? col[e] : -1;
      }
#pragma unroll
      for (int j = 0; j < kTileLoads; ++j) {
        const int64_t e = e0 + 32 * j + lane;
        const int64_t x = tile.r0 + tile.row_of(e);
        if (y[j] <= x || y[j] >= n) continue;   // as k_scan_rows counted
        const int64_t slot = static_cast<int64_t>(atomicAdd(&cur[y[j] >> sh], 1ull));
        if (slot < cap) part[slot] = make_int2(static_cast<int32_t>(x), y[j]);
        else latch(err, kErrValidate);
      }
    }
  }
}

// K searches for key[j] among the first ly[j] entries of row[j] (strictly
// increasing, below top[j] > key[j]), in lockstep, so that K loads are in
// flight per step: a single search is a chain of dependent reads.  The first
// probe is where the key would be in an evenly spread row, the next two around
// it: neighbours share the sector, the far probes of a plain binary search do
// not; then halving, which bounds the search for any row.  Not found: latched.
template <int K>
__device__ __forceinline__ void find_all(const int32_t* const (&row)[K], const int32_t (&key)[K], const int (&ly)[K],
                                         const int32_t (&top)[K], int32_t* err) {
  int lo[K], hi[K];
#pragma unroll
  for (int j = 0; j < K; ++j) {
    lo[j] = 0;
    hi[j] = ly[j];
  }
  for (int round = 0;; ++round) {
    bool more = false;
#pragma unroll
    for (int j = 0; j < K; ++j) {
      if (lo[j] < hi[j]) {
        more = true;
        int mid = (lo[j] + hi[j]) >> 1;
        if (round == 0)
          mid = static_cast<int>(static_cast<uint64_t>(static_cast<uint32_t>(key[j])) * ly[j] / static_cast<uint32_t>(top[j]));
        else if (round <= 2)
          mid = lo[j] > 0 && hi[j] == ly[j] ? min(lo[j] + 3, hi[j] - 1) : lo[j] == 0 && hi[j] < ly[j] ? max(hi[j] - 4, 0) : mid;
        if (row[j][mid] < key[j]) lo[j] = mid + 1;
        else hi[j] = mid;
      }
    }
    if (!more) break;
  }
#pragma unroll
  for (int j = 0; j < K; ++j)
    if (ly[j] > 0 && (lo[j] >= ly[j] || row[j][lo[j]] != key[j])) latch(err, kErrValidate);
}

// Every partitioned (x, y) found in L_y.
constexpr int kSearchLanes = 8;
__global__ void k_vcheck(int64_t n, const int64_t* __restrict__ rp, const int32_t* __restrict__ col,
                         const int32_t* __restrict__ low, const int2* __restrict__ part, int64_t total,
                         int32_t* err) {
  const int64_t stride = int64_t(gridDim.x) * blockDim.x * kSearchLanes;
  for (int64_t i0 = (blockIdx.x * int64_t(blockDim.x) + threadIdx.x) * kSearchLanes; i0 < total; i0 += stride) {
    const int32_t* row[kSearchLanes];
    int32_t key[kSearchLanes], top[kSearchLanes];
    int ly[kSearchLanes];
#pragma unroll
    for (int j = 0; j < kSearchLanes; ++j) {
      ly[j] = 0;
      key[j] = 0;
      top[j] = 1;
      row[j] = col;
      if (i0 + j >= total) continue;
      const int2 p = part[i0 + j];
      if (p.x < 0 || p.y <= p.x || p.y >= n) {   // a slot no valid entry wrote (malformed input)
        latch(err, kErrValidate);
        continue;
      }
      row[j] = col + rp[p.y];
      key[j] = p.x;
      top[j] = p.y;
      ly[j] = low[p.y];
      if (ly[j] == 0) latch(err, kErrValidate);   // nothing below the diagonal to find x in
    }
    find_all<kSearchLanes>(row, key, ly, top, err);
  }
}

// The same without the partition, for small graphs: every upper entry of a
// tile searched where it stands.
__global__ void __launch_bounds__(256) k_vdirect(int64_t n, const int64_t* __restrict__ rp,
                                                 const int32_t* __restrict__ col, int per, int split,
                                                 const int32_t* __restrict__ low, int32_t* err) {
  const int64_t tiles = (n + per - 1) / per, nw = int64_t(gridDim.x) * (blockDim.x >> 5);
  for (int64_t i = (blockIdx.x * int64_t(blockDim.x) + threadIdx.x) >> 5; i < tiles * split; i += nw) {
    const RowTile tile(rp, n, per * (i / split), per);
    for (int64_t e0 = tile.begin() + 32 * kTileLoads * (i % split); e0 < tile.end; e0 += 32 * kTileLoads * split) {
      const int32_t* row[kTileLoads];
      int32_t key[kTileLoads], top[kTileLoads];
      int ly[kTileLoads];
#pragma unroll
      for (int j = 0; j < kTileLoads; ++j) {
        const int64_t e = e0 + 32 * j + tile.lane;
        const int32_t x = static_cast<int32_t>(tile.r0 + tile.row_of(e)), y = e < tile.end ? col[e] : -1;
        const bool above = y > x && y < n;
        row[j] = above ? col + rp[y] : col;
        key[j] = above ? x : 0;
        top[j] = above ? y : 1;
        ly[j] = above ? low[y] : 0;
        if (above && ly[j] == 0) latch(err, kErrValidate);
      }
      find_all<kTileLoads>(row, key, ly, top, err);
    }
  }
}

// dst row q <- src row rowmap[q], values mapped through valmap, order kept;
// one warp per tile of `per` dst rows.
__global__ void __launch_bounds__(256) k_relabel(RowArgs a, int per, int split) {
  const int64_t tiles = (a.nrows + per - 1) / per, nw = int64_t(gridDim.x) * (blockDim.x >> 5);
  for (int64_t i = (blockIdx.x * int64_t(blockDim.x) + threadIdx.x) >> 5; i < tiles * split; i += nw) {
    const RowTile tile(a.dst_rp, a.nrows, per * (i / split), per);
    const int64_t q = tile.r0 + tile.lane;
    const bool own = tile.lane < per && q < a.nrows;
    const int64_t x = own ? (a.rowmap ? a.rowmap[q] : q) : 0;
    const int64_t from = own ? a.src_rp[x] - tile.off : 0;   // src entry of dst entry e: from + e
    if (own && a.src_rp[x + 1] - a.src_rp[x] != a.dst_rp[q + 1] - tile.off) latch(a.err, kErrRowLength);
    if (__any_sync(kFull, own && a.src_rp[x + 1] - a.src_rp[x] != a.dst_rp[q + 1] - tile.off)) continue;
    for (int64_t e0 = tile.begin() + 32 * kTileLoads * (i % split); e0 < tile.end; e0 += 32 * kTileLoads * split) {
      int32_t v[kTileLoads];
#pragma unroll
      for (int j = 0; j < kTileLoads; ++j) {
        const int64_t e = e0 + 32 * j + tile.lane;
        const int64_t f = __shfl_sync(kFull, from, tile.row_of(e));
        v[j] = e < tile.end ? a.src_col[f + e] : 0;
      }
#pragma unroll
      for (int j = 0; j < kTileLoads; ++j) {
        const int64_t e = e0 + 32 * j + tile.lane;
        if (e < tile.end) a.dst_col[e] = a.valmap ? a.valmap[v[j]] : v[j];
      }
    }
  }
}

// ---- canonical export: only the entries above the diagonal are sorted
//
// k_above_rows takes every position's row to node ids and keeps the entries
// above the diagonal, compacted at the start of the node's id-space row; their
// counts are scanned; then rows of up to kSortWarp such entries are sorted in a
// warp's registers and longer ones, listed, in shared memory.  n=2^25 (1.0e9
// pairs): relabelling, counting, compacting and sorting in separate passes over
// all entries, with the long rows found by scanning every row's count in every
// CTA, took 139 ms.

constexpr int kSortWarp = 256;      // one warp, 1 to 8 keys per lane
constexpr int kSortMid = 1024;      // listed, one warp per row, 16 or 32 keys per lane
constexpr int kSortKeys = 16;       // keys per thread of a CTA's sort
constexpr int kSortLists = 4;       // lists: up to kSortMid, 2048 (128 threads), 8192 (512), longer (1024)
constexpr int kSortBig = 1024 * kSortKeys;   // longer: a global slice

struct AboveArgs {
  int64_t n;
  const int64_t* rp;        // id-space offsets
  const int32_t* col;       // compacted rows
  int32_t* cnt;
  const int64_t* off;       // first pair of each row
  const Seg* segs;
  const int32_t* seg_of;
  int32_t* pairs;
  bool wide;                // pairs is 8-byte aligned: a pair per store (a caller's buffer may not be)
  int32_t* lists;           // rows with more than kSortWarp entries, by size (pair_lists.cuh, n places)
  unsigned long long* list_n;
};

__device__ __forceinline__ void put_pair(const AboveArgs& a, int64_t i, int32_t x, int32_t y) {
  if (a.wide) {
    reinterpret_cast<int2*>(a.pairs)[i] = make_int2(x, y);
  } else {
    a.pairs[2 * i] = x;
    a.pairs[2 * i + 1] = y;
  }
}
__device__ __forceinline__ void above_done(const AboveArgs& a, int64_t x, int c) {
  a.cnt[x] = c;
  if (c > kSortWarp) {
    const int k = c <= kSortMid ? 0 : c <= 128 * kSortKeys ? 1 : c <= 512 * kSortKeys ? 2 : 3;
    a.lists[pair_place(k, static_cast<int64_t>(atomicAdd(a.list_n + k, 1ull)), a.n)] = static_cast<int32_t>(x);
  }
}

// One warp per tile of `per` positions.
__global__ void __launch_bounds__(256) k_above_rows(AboveArgs a, const int64_t* __restrict__ src_rp,
                                                    const int32_t* __restrict__ src, const int32_t* __restrict__ order,
                                                    int32_t* __restrict__ dst, int per) {
  const int lane = threadIdx.x & 31;
  const int64_t tiles = (a.n + per - 1) / per, nw = int64_t(gridDim.x) * (blockDim.x >> 5);
  for (int64_t t = (blockIdx.x * int64_t(blockDim.x) + threadIdx.x) >> 5; t < tiles; t += nw) {
    const RowTile tile(src_rp, a.n, per * t, per);
    const bool own = lane < per && tile.r0 + lane < a.n;
    const int32_t x = own ? order[tile.r0 + lane] : 0;   // this lane's node
    const int64_t d0 = own ? a.rp[x] : 0;                // and its id-space row
    int c = 0;                                           // its entries kept so far
    for (int64_t e0 = tile.begin(); e0 < tile.end; e0 += 32 * kTileLoads) {
      int32_t y[kTileLoads];
#pragma unroll
      for (int j = 0; j < kTileLoads; ++j) {
        const int64_t e = e0 + 32 * j + lane;
        y[j] = e < tile.end ? src[e] : -1;
      }
#pragma unroll
      for (int j = 0; j < kTileLoads; ++j) y[j] = y[j] >= 0 ? order[y[j]] : -1;
#pragma unroll
      for (int j = 0; j < kTileLoads; ++j) {
        const int64_t eb = e0 + 32 * j;
        const int k = tile.row_of(eb + lane);
        const int32_t xr = __shfl_sync(kFull, x, k);
        const bool keep = y[j] > xr;   // (-1 past the end)
        const unsigned kept = __ballot_sync(kFull, keep);
        // lanes of the same row before this one: from the row's first entry on
        const int64_t o = __shfl_sync(kFull, tile.off, k);
        const int s0 = o > eb ? static_cast<int>(o - eb) : 0;
        const unsigned mine = kept & ((1u << lane) - 1u) & ~((1u << s0) - 1u);
        const int base = __shfl_sync(kFull, c, k);
        const int64_t d = __shfl_sync(kFull, d0, k);
        if (keep) dst[d + base + __popc(mine)] = y[j];
        c += own_count(tile, eb, kept);
      }
    }
    if (own) above_done(a, x, c);
  }
}

// Ascending sort of 32 K keys, key k of lane l having index 32 k + l.
template <int K>
__device__ __forceinline__ void warp_sort(int32_t (&v)[K]) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int size = 2; size <= 32 * K; size <<= 1) {
#pragma unroll
    for (int j = size >> 1; j > 0; j >>= 1) {
      if (j >= 32) {
#pragma unroll
        for (int k = 0; k < K; ++k) {
          const int l = k ^ (j >> 5);
          if (l > k) {
            const bool up = ((32 * k) & size) == 0;
            const int32_t a = min(v[k], v[l]), b = max(v[k], v[l]);
            v[k] = up ? a : b;
            v[l] = up ? b : a;
          }
        }
      } else {
#pragma unroll
        for (int k = 0; k < K; ++k) {
          const int32_t o = __shfl_xor_sync(kFull, v[k], j);
          const bool up = ((32 * k + lane) & size) == 0;
          v[k] = ((lane & j) == 0) == up ? min(v[k], o) : max(v[k], o);
        }
      }
    }
  }
}

// Row x's c kept entries (at base) sorted and written as pairs local to x's graph.
template <int K>
__device__ __forceinline__ void write_sorted(const AboveArgs& a, int32_t x, int64_t base, int c, int64_t o, int32_t sb) {
  const int lane = threadIdx.x & 31;
  int32_t v[K];
#pragma unroll
  for (int k = 0; k < K; ++k) v[k] = 32 * k + lane < c ? a.col[base + 32 * k + lane] : 0x7fffffff;
  warp_sort<K>(v);
#pragma unroll
  for (int k = 0; k < K; ++k)
    if (32 * k + lane < c) put_pair(a, o + 32 * k + lane, x - sb, v[k] - sb);
}

// Rows of at most kSortWarp kept entries, one warp per `per` rows (their counts
// and offsets loaded together).
__global__ void __launch_bounds__(256) k_above_warp(AboveArgs a, int per) {
  const int lane = threadIdx.x & 31;
  const int64_t tiles = (a.n + per - 1) / per, nw = int64_t(gridDim.x) * (blockDim.x >> 5);
  for (int64_t t = (blockIdx.x * int64_t(blockDim.x) + threadIdx.x) >> 5; t < tiles; t += nw) {
    const int64_t xl = per * t + lane;
    const bool own = lane < per && xl < a.n;
    const int cl = own ? a.cnt[xl] : 0;
    const int64_t bl = own ? a.rp[xl] : 0, ol = own ? a.off[xl] : 0;
    const int32_t sl = own && a.seg_of ? static_cast<int32_t>(a.segs[a.seg_of[xl]].off) : 0;
    for (unsigned left = __ballot_sync(kFull, cl > 0 && cl <= kSortWarp); left; left &= left - 1u) {
      const int r = __ffs(left) - 1;
      const int c = __shfl_sync(kFull, cl, r);
      const int64_t b = __shfl_sync(kFull, bl, r), o = __shfl_sync(kFull, ol, r);
      const int32_t sb = __shfl_sync(kFull, sl, r), x = static_cast<int32_t>(per * t + r);
      if (c <= 32) write_sorted<1>(a, x, b, c, o, sb);
      else if (c <= 64) write_sorted<2>(a, x, b, c, o, sb);
      else if (c <= 128) write_sorted<4>(a, x, b, c, o, sb);
      else write_sorted<8>(a, x, b, c, o, sb);
    }
  }
}

// The first list (more than kSortWarp, at most kSortMid kept entries), one warp
// per row: spread over all warps, where the tiles would leave a few warps
// with most of the work.  (256 threads per row in shared memory, up to 2048
// entries, took 17.4 ms at n=2^25.)
__global__ void __launch_bounds__(256) k_above_listed(AboveArgs a) {
  const int64_t rows = static_cast<int64_t>(a.list_n[0]), nw = int64_t(gridDim.x) * (blockDim.x >> 5);
  for (int64_t i = (blockIdx.x * int64_t(blockDim.x) + threadIdx.x) >> 5; i < rows; i += nw) {
    const int32_t x = a.lists[pair_place(0, i, a.n)];
    const int c = a.cnt[x];
    const int32_t sb = a.seg_of ? static_cast<int32_t>(a.segs[a.seg_of[x]].off) : 0;
    if (c <= 512) write_sorted<16>(a, x, a.rp[x], c, a.off[x], sb);
    else write_sorted<32>(a, x, a.rp[x], c, a.off[x], sb);
  }
}

// Ascending sort of up to kSortKeys NT keys held kSortKeys per thread (warp w,
// key k, lane l: index 512 w + 32 k + l), P a power of two, 512 <= P: strides
// below 512 stay in a warp's registers, the others (15 of 105 steps at 16384
// keys) go through shared memory.  A bitonic sort that does every step in
// shared memory took 19.9 ms for the rows above 1024 entries at n=2^25, this 8.6.
template <int NT>
__device__ void cta_sort(int32_t (&v)[kSortKeys], int32_t* buf, int P) {
  constexpr int K = kSortKeys;
  const int lane = threadIdx.x & 31, at = (threadIdx.x >> 5) * 32 * K + lane;
  for (int size = 2; size <= P; size <<= 1) {
    for (int j = size >> 1; j >= 32 * K; j >>= 1) {
      __syncthreads();
#pragma unroll
      for (int k = 0; k < K; ++k) buf[at + 32 * k] = v[k];
      __syncthreads();
      const bool up = (at & size) == 0, low = (at & j) == 0;   // the same for the warp's keys
#pragma unroll
      for (int k = 0; k < K; ++k) {
        const int32_t o = buf[(at + 32 * k) ^ j];
        v[k] = low == up ? min(v[k], o) : max(v[k], o);
      }
    }
#pragma unroll
    for (int jj = 16 * K; jj >= 32; jj >>= 1) {   // across a lane's keys
      if (jj >= size) continue;
#pragma unroll
      for (int k = 0; k < K; ++k) {
        const int l = k ^ (jj >> 5);
        if (l > k) {
          const bool up = ((at + 32 * k) & size) == 0;
          const int32_t a = min(v[k], v[l]), b = max(v[k], v[l]);
          v[k] = up ? a : b;
          v[l] = up ? b : a;
        }
      }
    }
    for (int j = size > 32 ? 16 : size >> 1; j > 0; j >>= 1) {   // across lanes
#pragma unroll
      for (int k = 0; k < K; ++k) {
        const int32_t o = __shfl_xor_sync(kFull, v[k], j);
        const bool up = ((at + 32 * k) & size) == 0;
        v[k] = ((lane & j) == 0) == up ? min(v[k], o) : max(v[k], o);
      }
    }
  }
}

// The rows of a list, one CTA each: up to kSortKeys NT entries in registers,
// more (the last list only) in a global slice per CTA.
template <int NT>
__global__ void __launch_bounds__(NT, NT == 1024 ? 1 : 1024 / NT) k_above_block(AboveArgs a, int which, int32_t* gws, int64_t slice) {
  __shared__ int32_t buf[kSortKeys * NT > 12288 ? 1 : kSortKeys * NT];
  extern __shared__ int32_t dbuf[];
  __shared__ int64_t red[BlockTeam<NT>::kRedSlots];
  int32_t* const b0 = kSortKeys * NT > 12288 ? dbuf : buf;
  const int lane = threadIdx.x & 31, at = (threadIdx.x >> 5) * 32 * kSortKeys + lane;
  const int64_t rows = static_cast<int64_t>(a.list_n[which]);
  for (int64_t i = blockIdx.x; i < rows; i += gridDim.x) {
    const int32_t x = a.lists[pair_place(which, i, a.n)];
    const int c = a.cnt[x];
    const int64_t b = a.rp[x], o = a.off[x];
    const int32_t sb = a.seg_of ? static_cast<int32_t>(a.segs[a.seg_of[x]].off) : 0;
    const int P = next_pow2(c);
    if (c <= kSortKeys * NT) {
      int32_t v[kSortKeys];
#pragma unroll
      for (int k = 0; k < kSortKeys; ++k) v[k] = at + 32 * k < c ? a.col[b + at + 32 * k] : 0x7fffffff;
      cta_sort<NT>(v, b0, P);
#pragma unroll
      for (int k = 0; k < kSortKeys; ++k)
        if (at + 32 * k < c) put_pair(a, o + at + 32 * k, x - sb, v[k] - sb);
    } else {
      BlockTeam<NT> tm(red);
      int32_t* g = gws + slice * blockIdx.x;
      for (int q = threadIdx.x; q < P; q += NT) g[q] = q < c ? a.col[b + q] : 0x7fffffff;
      tm.sync();
      team_bitonic_sort(tm, g, P);
      for (int q = threadIdx.x; q < c; q += NT) put_pair(a, o + q, x - sb, g[q] - sb);
    }
    __syncthreads();
  }
}

unsigned grid_of(int64_t work, int threads, int num_sms) {
  const int64_t want = (work + threads - 1) / threads;
  const int64_t cap = int64_t(num_sms) * 16;
  return static_cast<unsigned>(std::max<int64_t>(1, std::min(want, cap)));
}

}  // namespace

int permute_rows(Graph* h, int64_t nrows, const int64_t* src_rp, const int32_t* src_col,
                 const int32_t* rowmap, const int32_t* valmap, const int64_t* dst_rp, int32_t* dst_col) {
  if (nrows == 0) return CB_OK;
  RowArgs a{nrows, src_rp, src_col, rowmap, valmap, dst_rp, dst_col, h->err};
  const unsigned wgrid = grid_of(nrows, 8, h->num_sms);
  k_rows_warp<<<wgrid, 256, 0, h->stream>>>(a);
  CB_CUDA(h, cudaGetLastError());
  ++h->launches;
  if (h->maxdeg > kRowWarpMax) {
    // global slice per CTA for rows longer than the shared-memory buffer
    int64_t slice = 0;
    int ctas = h->num_sms * 2;
    int32_t* gws = nullptr;
    if (h->maxdeg > kRowBlockSmem) {
      slice = next_pow2_host(h->maxdeg);
      const size_t budget = h->ws_slice * static_cast<size_t>(h->ws_ctas);
      ctas = static_cast<int>(std::max<int64_t>(1, std::min<int64_t>(ctas, budget / (slice * 4))));
      if (budget < static_cast<size_t>(slice) * 4) return fail(h, CB_ENOMEM, "row workspace too small");
      gws = static_cast<int32_t*>(h->ws_global);
    }
    CB_CUDA(h, cudaFuncSetAttribute(k_rows_block, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                    kRowBlockSmem * 4));
    k_rows_block<<<ctas, 256, kRowBlockSmem * 4, h->stream>>>(a, gws, slice);
    CB_CUDA(h, cudaGetLastError());
  ++h->launches;
  }
  return CB_OK;
}

// Up to this many bytes of adjacency the symmetry is checked in place.  At
// n=2^17 (24 MB) the searches all over L2 take 141 us against 132 for scan,
// partition and check, but an allocation and four launches fewer: 0.70 against
// 0.77 ms for the whole creation.
constexpr int64_t kDirectBytes = int64_t(32) << 20;

int scan_rows(Graph* h, const int64_t* rp, const int32_t* col, int64_t n, Validation* v) {
  cudaStream_t s = h->stream;
  unsigned long long* found = reinterpret_cast<unsigned long long*>(h->scratch);
  int32_t* low = h->pos[1];   // not in use before the first super step
  if (n) {
    CB_CUDA(h, cudaMemsetAsync(found + 1, 0, (kScanWords - 1) * sizeof(unsigned long long), s));
    if (h->nnz * 4 <= kDirectBytes) {
      const int per = rows_per_warp(n, h->num_sms);
      k_scan_rows<false><<<grid_of((n + per - 1) / per * 32, kVThreads, h->num_sms), kVThreads, 0, s>>>(
          n, rp, col, per, 0, 0, nullptr, low, found, h->err);
    } else {
      if (!v->ws) {
        while (((n - 1) >> v->sh) >= kVBuckets) ++v->sh;
        v->nb = static_cast<int>(((n - 1) >> v->sh) + 1);
        v->ctas = static_cast<int>(std::max<int64_t>(1, std::min<int64_t>(h->num_sms * 4, (n + 511) / 512)));
        const int64_t cells = int64_t(v->nb) * v->ctas;
        const size_t place = (sizeof(int32_t) * cells + 31) & ~size_t(31), scan = place + sizeof(int64_t) * (cells + 1);
        v->bytes = scan + scan_ws_bytes(cells);
        CB_CUDA(h, dev_alloc(h, reinterpret_cast<void**>(&v->ws), v->bytes));
        v->counts = reinterpret_cast<int32_t*>(v->ws);
        v->place = reinterpret_cast<int64_t*>(v->ws + place);
        v->scan = v->ws + scan;
      }
      k_scan_rows<true><<<v->ctas, kVThreads, 0, s>>>(n, rp, col, 32, v->sh, v->nb, v->counts, low, found, h->err);
    }
    CB_CUDA(h, cudaGetLastError());
    ++h->launches;
  }
  // the error word and the scratch words lie next to each other
  struct {
    int32_t err[64];
    int64_t found[kScanWords];
  } got;
  static_assert(sizeof(got.err) == 256, "the scratch follows the error word's 256 bytes");
  CB_CUDA(h, cudaMemcpyAsync(&got, h->err, sizeof(got), cudaMemcpyDeviceToHost, s));
  CB_CUDA(h, cudaStreamSynchronize(s));
  v->err = got.err[0];
  v->maxdeg = got.found[kScanMaxdeg];
  v->unsorted = got.found[kScanUnsorted] != 0;
  v->bad = got.found[kScanBad] != 0;
  v->upper = got.found[kScanUpper];
  v->lower = got.found[kScanLower];
  return CB_OK;
}

void free_validation(Graph* h, Validation* v) {
  if (!v->ws) return;
  cudaFreeAsync(v->ws, h->stream);
  h->dev_bytes -= static_cast<int64_t>(v->bytes);
  v->ws = nullptr;
}

int validate_sorted_graph(Graph* h, const int64_t* rp, const int32_t* col, int64_t n, Validation* v,
                          int32_t* grouped) {
  if (n == 0) return CB_OK;
  cudaStream_t s = h->stream;
  const int32_t* low = h->pos[1];
  if (!v->ws) {
    const int per = rows_per_warp(n, h->num_sms);
    k_vdirect<<<grid_of((n + per - 1) / per * 32 * tile_split(per), 256, h->num_sms), 256, 0, s>>>(n, rp, col, per,
                                                                                                     tile_split(per), low, h->err);
    CB_CUDA(h, cudaGetLastError());
    ++h->launches;
    return CB_OK;
  }
  const int64_t cells = int64_t(v->nb) * v->ctas;
  CB_CUDA(h, exclusive_scan_i32(v->counts, v->place, cells, v->scan, s, &h->launches));
  // as many entries above the diagonal as below, so they are half: `grouped`
  // holds row_ptr[n] int32
  const int64_t cap = h->nnz / 2;
  k_vpart<<<v->ctas, kVThreads, 0, s>>>(n, rp, col, v->sh, v->nb, v->place, reinterpret_cast<int2*>(grouped), cap,
                                        h->err);
  k_vcheck<<<grid_of(n, 256, h->num_sms), 256, 0, s>>>(n, rp, col, low, reinterpret_cast<const int2*>(grouped), cap,
                                                       h->err);
  CB_CUDA(h, cudaGetLastError());
  h->launches += 2;
  return CB_OK;
}

int relabel_rows(Graph* h, int64_t nrows, const int64_t* src_rp, const int32_t* src_col, const int32_t* rowmap,
                 const int32_t* valmap, const int64_t* dst_rp, int32_t* dst_col) {
  if (nrows == 0) return CB_OK;
  RowArgs a{nrows, src_rp, src_col, rowmap, valmap, dst_rp, dst_col, h->err};
  const int per = rows_per_warp(nrows, h->num_sms);
  k_relabel<<<grid_of((nrows + per - 1) / per * 32 * tile_split(per), 256, h->num_sms), 256, 0, h->stream>>>(a, per, tile_split(per));
  CB_CUDA(h, cudaGetLastError());
  ++h->launches;
  return CB_OK;
}

// Canonical pairs of the current step.
int export_sorted_pairs(Graph* h, int32_t* pairs) {
  const int64_t n = h->n;
  if (n == 0) return CB_OK;
  const int spare = 1 - h->cur;
  int32_t* cnt = h->pos[spare];    // free between super steps, as the offsets,
  int64_t* off = h->rp[spare];     // the spare adjacency and the class lists are
  cudaStream_t s = h->stream;
  AboveArgs a{};
  a.n = n;
  a.rp = h->rp_id;
  a.col = h->col[spare];
  a.cnt = cnt;
  a.off = off;
  a.segs = h->segs;
  a.seg_of = h->seg_of;
  a.pairs = pairs;
  a.wide = reinterpret_cast<uintptr_t>(pairs) % 8 == 0;
  a.lists = h->lists;   // kClassLists n / 2 places
  static_assert((kSortLists + 1) / 2 * 2 <= kClassLists, "");
  a.list_n = reinterpret_cast<unsigned long long*>(h->scratch);
  const bool lists = h->maxdeg > kSortWarp;
  if (lists) CB_CUDA(h, cudaMemsetAsync(a.list_n, 0, kSortLists * sizeof(unsigned long long), s));
  const int per = rows_per_warp(n, h->num_sms);
  const unsigned tgrid = grid_of((n + per - 1) / per * 32, 256, h->num_sms);
  k_above_rows<<<tgrid, 256, 0, s>>>(a, h->rp[h->cur], h->col[h->cur], h->order[h->cur], h->col[spare], per);
  CB_CUDA(h, cudaGetLastError());
  CB_CUDA(h, exclusive_scan_i32(cnt, off, n, h->scan_ws, s, &h->launches));
  k_above_warp<<<tgrid, 256, 0, s>>>(a, per);
  CB_CUDA(h, cudaGetLastError());
  h->launches += 2;
  if (lists) {
    k_above_listed<<<h->num_sms * 4, 256, 0, s>>>(a);
    CB_CUDA(h, cudaGetLastError());
    ++h->launches;
  }
  if (h->maxdeg > kSortMid) {
    k_above_block<128><<<h->num_sms * 8, 128, 0, s>>>(a, 1, nullptr, 0);
    CB_CUDA(h, cudaGetLastError());
    ++h->launches;
  }
  if (h->maxdeg > 128 * kSortKeys) {
    k_above_block<512><<<h->num_sms * 2, 512, 0, s>>>(a, 2, nullptr, 0);
    CB_CUDA(h, cudaGetLastError());
    ++h->launches;
  }
  if (h->maxdeg > 512 * kSortKeys) {
    int64_t slice = 0;
    int ctas = h->num_sms;
    int32_t* gws = nullptr;
    if (h->maxdeg > kSortBig) {
      slice = next_pow2_host(h->maxdeg);
      const size_t budget = h->ws_slice * static_cast<size_t>(h->ws_ctas);
      if (budget < static_cast<size_t>(slice) * 4) return fail(h, CB_ENOMEM, "row workspace too small");
      ctas = static_cast<int>(std::max<int64_t>(1, std::min<int64_t>(ctas, budget / (slice * 4))));
      gws = static_cast<int32_t*>(h->ws_global);
    }
    CB_CUDA(h, cudaFuncSetAttribute(k_above_block<1024>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSortBig * 4));
    k_above_block<1024><<<ctas, 1024, kSortBig * 4, s>>>(a, 3, gws, slice);
    CB_CUDA(h, cudaGetLastError());
    ++h->launches;
  }
  return CB_OK;
}

}  // namespace cb

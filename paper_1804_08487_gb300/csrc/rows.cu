// Row-level utilities outside the super step: relabelling a CSR into another
// row order and node numbering (with each row sorted), input validation, the
// inverse of a permutation and the canonical edge export (Section 2: ordered
// edges [a,b], a<b).
#include <algorithm>

#include "cb_internal.cuh"
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

__global__ void k_check_rp(int64_t n, const int64_t* __restrict__ rp, int32_t* err) {
  for (int64_t x = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; x < n; x += int64_t(gridDim.x) * blockDim.x) {
    const int64_t d = rp[x + 1] - rp[x];
    if (d < 0 || d >= n || (x == 0 && rp[0] != 0)) latch(err, kErrValidate);
  }
}

// Validation of sorted rows: strictly increasing, in range, no self loop,
// and symmetric.  Symmetry is checked exactly:
//   - every entry y > x of row x must be found among the entries of row y
//     below the diagonal (L_y);
//   - the entries above the diagonal, summed over all rows, must be as many
//     as those below.
// The found entries are distinct (rows are strictly increasing), so each L_y
// holds at least as many as point into it, and the totals force equality.
// For locality the upper entries are first partitioned into buckets of
// target rows, with one reservation per bucket and CTA. Each bucket's
// searches then stay within a few MB of rows that L2 holds.

constexpr int kVBuckets = 4096;     // target-row buckets of the partition

// low[x] = entries of row x below x (a lower bound in the sorted row)
__global__ void k_lower_count(int64_t n, const int64_t* __restrict__ rp, const int32_t* __restrict__ col,
                              int32_t* __restrict__ low) {
  for (int64_t x = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; x < n; x += int64_t(gridDim.x) * blockDim.x)
    low[x] = lower_bound(col + rp[x], static_cast<int>(rp[x + 1] - rp[x]), static_cast<int32_t>(x));
}

// The validation's partition: CTA c of kVCtas takes row tiles [c per, (c+1)
// per), counts its upper entries per bucket (k_vcount, with the row checks),
// and, after a scan over (bucket, CTA), writes them there (k_vpart).  Both
// passes read the entries once, as runs of 32 rows per warp.
constexpr int kVThreads = 512;

// flags[0]: some row is not strictly increasing; flags[1]: an id out of range
// or a self loop.
__global__ void __launch_bounds__(kVThreads) k_vcount(int64_t n, const int64_t* __restrict__ rp,
                                                      const int32_t* __restrict__ col, int sh, int nb,
                                                      int32_t* __restrict__ counts, int32_t* __restrict__ flags) {
  __shared__ int32_t cnt[kVBuckets];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int64_t tiles = (n + 31) / 32, per = (tiles + gridDim.x - 1) / gridDim.x;
  const int64_t t0 = blockIdx.x * per, t1 = t0 + per < tiles ? t0 + per : tiles;
  for (int b = threadIdx.x; b < nb; b += blockDim.x) cnt[b] = 0;
  __syncthreads();
  bool unsorted = false, bad = false;
  for (int64_t t = t0 + w; t < t1; t += kVThreads / 32) {
    const RowTile tile(rp, n, 32 * t);
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
        if (e >= tile.end) continue;
        const int64_t x = tile.r0 + k;
        const bool wrong = y[j] < 0 || y[j] >= n || y[j] == x;
        bad |= wrong;
        unsorted |= e > first && prev >= y[j];
        if (!wrong && y[j] > x) atomicAdd(&cnt[y[j] >> sh], 1);
      }
    }
  }
  if (__any_sync(kFull, unsorted) && lane == 0) flags[0] = 1;
  if (__any_sync(kFull, bad) && lane == 0) flags[1] = 1;
  __syncthreads();
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
        if (y[j] <= x || y[j] >= n) continue;   // as k_vcount counted
        const int64_t slot = static_cast<int64_t>(atomicAdd(&cur[y[j] >> sh], 1ull));
        if (slot < cap) part[slot] = make_int2(static_cast<int32_t>(x), y[j]);
        else latch(err, kErrValidate);
      }
    }
  }
}

// Every partitioned (x, y) found in L_y; and as many entries above the
// diagonal as below (*all_upper against the scan of low, grp[n]).
// A thread runs kSearchLanes binary searches in lockstep, so that many loads
// are in flight per step: a single search is a chain of dependent L2 reads.
constexpr int kSearchLanes = 8;

__global__ void k_vcheck(int64_t n, const int64_t* __restrict__ rp, const int32_t* __restrict__ col,
                         const int32_t* __restrict__ low, const int2* __restrict__ part,
                         const int64_t* __restrict__ all_upper, const int64_t* __restrict__ grp, int64_t cap,
                         int32_t* err) {
  const int64_t all = *all_upper;
  if (blockIdx.x == 0 && threadIdx.x == 0 && all != grp[n]) latch(err, kErrValidate);
  const int64_t total = all < cap ? all : cap;
  const int64_t stride = int64_t(gridDim.x) * blockDim.x * kSearchLanes;
  for (int64_t i0 = (blockIdx.x * int64_t(blockDim.x) + threadIdx.x) * kSearchLanes; i0 < total; i0 += stride) {
    const int32_t* row[kSearchLanes];
    int32_t key[kSearchLanes];
    int lo[kSearchLanes], hi[kSearchLanes], ly[kSearchLanes], top[kSearchLanes];
#pragma unroll
    for (int j = 0; j < kSearchLanes; ++j) {
      lo[j] = 0;
      hi[j] = 0;
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
      hi[j] = ly[j];
      lo[j] = 0;
      if (ly[j] == 0) latch(err, kErrValidate);   // nothing below the diagonal to find x in
    }
    // first probe where the key would be in an evenly spread row, then around
    // it: neighbours share the sector, the far probes of a plain binary search
    // do not; then halving, which bounds the search for any row
    for (int round = 0;; ++round) {
      bool more = false;
#pragma unroll
      for (int j = 0; j < kSearchLanes; ++j) {
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
    for (int j = 0; j < kSearchLanes; ++j)
      if (ly[j] > 0 && (lo[j] >= ly[j] || row[j][lo[j]] != key[j])) latch(err, kErrValidate);
  }
}

// dst row q <- src row rowmap[q], values mapped through valmap, order kept.
__global__ void k_relabel(RowArgs a) {
  const int lane = threadIdx.x & 31;
  const int64_t nw = int64_t(gridDim.x) * (blockDim.x >> 5);
  for (int64_t q = (blockIdx.x * int64_t(blockDim.x) + threadIdx.x) >> 5; q < a.nrows; q += nw) {
    const int64_t x = a.rowmap ? a.rowmap[q] : q;
    const int64_t s0 = a.src_rp[x], len = a.src_rp[x + 1] - s0;
    const int64_t d0 = a.dst_rp[q];
    if (len != a.dst_rp[q + 1] - d0) {
      if (lane == 0) latch(a.err, kErrRowLength);
      continue;
    }
    for (int64_t i = lane; i < len; i += 32) {
      const int32_t v = a.src_col[s0 + i];
      a.dst_col[d0 + i] = a.valmap ? a.valmap[v] : v;
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
constexpr int kSortBig = kRowBlockSmem;   // 1024 threads, 64 KB; longer: a global slice

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
  int32_t* list[2];         // rows with more than kSortWarp, kSortMid entries
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
    const int k = c > kSortMid ? 1 : 0;
    a.list[k][atomicAdd(a.list_n + k, 1ull)] = static_cast<int32_t>(x);
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
        // the owner's row covers lanes [off - eb, next - eb)
        const int64_t nx = __shfl_down_sync(kFull, tile.off, 1);
        const int64_t lo = tile.off - eb, hi = (lane == 31 ? tile.end : nx) - eb;
        if (hi > 0 && lo < 32) {
          const unsigned from = lo > 0 ? ~((1u << lo) - 1u) : ~0u;
          const unsigned to = hi < 32 ? (1u << hi) - 1u : ~0u;
          c += __popc(kept & from & to);
        }
      }
    }
    if (own) above_done(a, x, c);
  }
}

// Rows per warp of the export's kernels: 32, fewer where that would leave
// warps without rows (n=4096: 32 rows per warp took 85 us for the export, 4 rows 60).
int rows_per_warp(int64_t n, int num_sms) {
  int64_t r = 32;
  while (r > 4 && (n + r - 1) / r < int64_t(num_sms) * 16) r >>= 1;
  return static_cast<int>(r);
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
    const int32_t x = a.list[0][i];
    const int c = a.cnt[x];
    const int32_t sb = a.seg_of ? static_cast<int32_t>(a.segs[a.seg_of[x]].off) : 0;
    if (c <= 512) write_sorted<16>(a, x, a.rp[x], c, a.off[x], sb);
    else write_sorted<32>(a, x, a.rp[x], c, a.off[x], sb);
  }
}

// The second list's rows, one CTA each, in `cap` ints of shared memory or, above that, a
// global slice per CTA.
template <int NT>
__global__ void __launch_bounds__(NT) k_above_block(AboveArgs a, int cap, int32_t* gws, int64_t slice) {
  extern __shared__ int32_t sbuf[];
  __shared__ int64_t red[BlockTeam<NT>::kRedSlots];
  BlockTeam<NT> tm(red);
  const int64_t rows = static_cast<int64_t>(a.list_n[1]);
  for (int64_t i = blockIdx.x; i < rows; i += gridDim.x) {
    const int32_t x = a.list[1][i];
    const int c = a.cnt[x];
    const int64_t b = a.rp[x], o = a.off[x];
    const int32_t sb = a.seg_of ? static_cast<int32_t>(a.segs[a.seg_of[x]].off) : 0;
    int32_t* buf = c <= cap ? sbuf : gws + slice * blockIdx.x;
    const int P = next_pow2(c);
    for (int q = threadIdx.x; q < P; q += NT) buf[q] = q < c ? a.col[b + q] : 0x7fffffff;
    tm.sync();
    team_bitonic_sort(tm, buf, P);
    for (int q = threadIdx.x; q < c; q += NT) put_pair(a, o + q, x - sb, buf[q] - sb);
    tm.sync();
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

// The rows' checks and upper entries per bucket: a first pass over the
// entries that also says whether every row is strictly increasing
// (synchronises).  Its scratch, kept for validate_sorted_graph, is freed by
// free_validation.
int scan_rows(Graph* h, const int64_t* rp, const int32_t* col, int64_t n, Validation* v, bool* sorted) {
  *sorted = true;
  if (n == 0) return CB_OK;
  cudaStream_t s = h->stream;
  if (!v->ws) {
    v->sh = 0;
    while (((n - 1) >> v->sh) >= kVBuckets) ++v->sh;
    v->nb = static_cast<int>(((n - 1) >> v->sh) + 1);
    v->ctas = static_cast<int>(std::max<int64_t>(1, std::min<int64_t>(h->num_sms * 4, (n + 511) / 512)));
    const int64_t cells = int64_t(v->nb) * v->ctas;
    const size_t place = (sizeof(int32_t) * cells + 63) & ~size_t(31), scan = place + sizeof(int64_t) * (cells + 1);
    v->bytes = scan + scan_ws_bytes(cells);
    CB_CUDA(h, dev_alloc(h, reinterpret_cast<void**>(&v->ws), v->bytes));
    v->counts = reinterpret_cast<int32_t*>(v->ws) + 4;
    v->flags = reinterpret_cast<int32_t*>(v->ws);
    v->place = reinterpret_cast<int64_t*>(v->ws + place);
    v->scan = v->ws + scan;
  }
  CB_CUDA(h, cudaMemsetAsync(v->flags, 0, 2 * sizeof(int32_t), s));
  k_vcount<<<v->ctas, kVThreads, 0, s>>>(n, rp, col, v->sh, v->nb, v->counts, v->flags);
  CB_CUDA(h, cudaGetLastError());
  ++h->launches;
  int32_t f[2] = {0, 0};
  CB_CUDA(h, cudaMemcpyAsync(f, v->flags, sizeof(f), cudaMemcpyDeviceToHost, s));
  CB_CUDA(h, cudaStreamSynchronize(s));
  *sorted = f[0] == 0;
  v->bad = f[1] != 0;
  return CB_OK;
}

void free_validation(Graph* h, Validation* v) {
  if (!v->ws) return;
  cudaFreeAsync(v->ws, h->stream);
  h->dev_bytes -= static_cast<int64_t>(v->bytes);
  v->ws = nullptr;
}

// Rows that scan_rows found well formed: symmetric, or kErrValidate latched
// (not synchronising).
int validate_sorted_graph(Graph* h, const int64_t* rp, const int32_t* col, int64_t n, Validation* v,
                          int32_t* grouped) {
  if (n == 0) return CB_OK;
  cudaStream_t s = h->stream;
  // scratch: low in a step buffer of n int32, its scan in rp[1] (n+1 int64),
  // none in use before the first super step; the partition in `grouped`
  int32_t* low = h->pos[1];
  int64_t* grp = h->rp[1];
  const unsigned g = grid_of(n, 256, h->num_sms);
  const int64_t cells = int64_t(v->nb) * v->ctas;
  k_lower_count<<<g, 256, 0, s>>>(n, rp, col, low);
  CB_CUDA(h, exclusive_scan_i32(low, grp, n, h->scan_ws, s, &h->launches));
  CB_CUDA(h, exclusive_scan_i32(v->counts, v->place, cells, v->scan, s, &h->launches));
  // the scratch holds row_ptr[n] int32: room for row_ptr[n] / 2 pairs,
  // exactly the entries above the diagonal of a symmetric graph
  const int64_t cap = h->nnz / 2;
  k_vpart<<<v->ctas, kVThreads, 0, s>>>(n, rp, col, v->sh, v->nb, v->place, reinterpret_cast<int2*>(grouped), cap,
                                        h->err);
  k_vcheck<<<g, 256, 0, s>>>(n, rp, col, low, reinterpret_cast<const int2*>(grouped), v->place + cells, grp, cap, h->err);
  CB_CUDA(h, cudaGetLastError());
  h->launches += 3;
  return CB_OK;
}

int relabel_rows(Graph* h, int64_t nrows, const int64_t* src_rp, const int32_t* src_col, const int32_t* rowmap,
                 const int32_t* valmap, const int64_t* dst_rp, int32_t* dst_col) {
  if (nrows == 0) return CB_OK;
  RowArgs a{nrows, src_rp, src_col, rowmap, valmap, dst_rp, dst_col, h->err};
  k_relabel<<<grid_of(nrows * 32, 256, h->num_sms), 256, 0, h->stream>>>(a);
  CB_CUDA(h, cudaGetLastError());
  ++h->launches;
  return CB_OK;
}

int check_row_offsets(Graph* h, const int64_t* rp, int64_t n) {
  if (n == 0) return CB_OK;
  k_check_rp<<<grid_of(n, 256, h->num_sms), 256, 0, h->stream>>>(n, rp, h->err);
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
  a.list[0] = h->lists;
  a.list[1] = h->lists + n;
  a.list_n = reinterpret_cast<unsigned long long*>(h->counters) + 2 * kCounters + 2;
  const bool lists = h->maxdeg > kSortWarp;
  if (lists) CB_CUDA(h, cudaMemsetAsync(a.list_n, 0, 2 * sizeof(unsigned long long), s));
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
    int64_t slice = 0;
    int ctas = h->num_sms * 2;
    int32_t* gws = nullptr;
    if (h->maxdeg > kSortBig) {
      slice = next_pow2_host(h->maxdeg);
      const size_t budget = h->ws_slice * static_cast<size_t>(h->ws_ctas);
      if (budget < static_cast<size_t>(slice) * 4) return fail(h, CB_ENOMEM, "row workspace too small");
      ctas = static_cast<int>(std::max<int64_t>(1, std::min<int64_t>(ctas, budget / (slice * 4))));
      gws = static_cast<int32_t*>(h->ws_global);
    }
    const int cap = static_cast<int>(std::min<int64_t>(kSortBig, next_pow2_host(h->maxdeg)));
    CB_CUDA(h, cudaFuncSetAttribute(k_above_block<1024>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSortBig * 4));
    k_above_block<1024><<<ctas, 1024, cap * 4, s>>>(a, cap, gws, slice);
    CB_CUDA(h, cudaGetLastError());
    ++h->launches;
  }
  return CB_OK;
}

}  // namespace cb

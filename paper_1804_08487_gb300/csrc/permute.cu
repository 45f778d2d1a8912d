// The permutation pi of a super step (Def. "Undirected Global Trade"): node x
// gets the key philox64(seed; x, 0, g, 0) and the nodes are ordered by
// (key, x).  Keys are uniform, so an MSD bucket sort does it: buckets by the
// top B key bits (about 512 to 1023 nodes each), each sorted by one CTA in
// shared memory by a counting sort on the 10 key bits below the highest bit
// where the bucket's keys differ (about one key per bin; keys sharing a bin
// are ranked against each other).  The same kernels write the row offsets of
// the new order and build the size-class lists of the current step's trades
// (classes.cuh), so a super step spends one or two launches before its trades:
//   - small handles: k_perm_rescan, one CTA per bucket, which computes every
//     key of its graph and keeps those of its bucket; the others only count
//     towards the bucket's first position and row offset;
//   - larger ones: k_perm_scatter puts the node ids into their buckets (one
//     64-bit atomic per node: bucket fill and degree sum), its last CTA scans
//     the buckets, and k_bucket_sort sorts them (keys computed again: cheaper
//     than 16 bytes per node of traffic).
// Buckets that exceed their space or the shared memory ("bucket_cap") are
// ranked by a slow path that needs neither.
#include "cb_internal.cuh"
#include "classes.cuh"
#include "philox.cuh"
#include "team.cuh"

#include <algorithm>
#include <cmath>
#include <mutex>

namespace cb {

int bucket_bits(int64_t n) {
  int lg = 0;
  while ((int64_t(1) << (lg + 1)) <= n) ++lg;
  return lg > 9 ? lg - 9 : 0;
}

// Space of one bucket of a graph of `span` nodes in 2^B buckets: the mean and
// twelve standard deviations.
int64_t bucket_space(int64_t span, int B) {
  if (B == 0) return span;
  const int64_t mean = (span >> B) + 1;
  return std::min<int64_t>(span, mean + 12 * (static_cast<int64_t>(std::sqrt(static_cast<double>(mean))) + 1) + 64);
}

namespace {

constexpr int kPermThreads = 256;

__device__ __forceinline__ uint32_t bucket_of(uint64_t key, int B) {
  return B == 0 ? 0u : static_cast<uint32_t>(key >> (64 - B));
}

// Where node keys come from: a handle's segment table (each segment at its
// device step + dg, or every segment at g_abs when use_abs), or one segment
// passed by value (segs == nullptr).
struct KeySrc {
  const Seg* segs;
  const int32_t* seg_of;
  Seg s0;
  uint32_t dg;
  int use_abs;
  uint32_t g_abs;
};

// One graph's part of it.  (__ldg for what creation fixed; the step counter is
// written by the end of each step, see after_previous().)
struct SegKey {
  uint64_t seed;
  int64_t off, n, span, base, slot_base;
  uint32_t g;
  int B, cap;
};
__device__ __forceinline__ SegKey seg_key(const KeySrc& ks, int i) {
  const Seg* S = ks.segs ? ks.segs + i : nullptr;
  SegKey k;
  k.seed = S ? __ldg(&S->seed) : ks.s0.seed;
  k.off = S ? __ldg(&S->off) : ks.s0.off;
  k.n = S ? __ldg(&S->n) : ks.s0.n;
  k.span = S ? __ldg(&S->span) : ks.s0.span;
  k.base = S ? __ldg(&S->bucket_base) : ks.s0.bucket_base;
  k.slot_base = S ? __ldg(&S->slot_base) : ks.s0.slot_base;
  k.g = ks.use_abs ? ks.g_abs : (S ? S->g : ks.s0.g) + ks.dg;
  k.B = S ? __ldg(&S->B) : ks.s0.B;
  k.cap = S ? __ldg(&S->cap) : ks.s0.cap;
  return k;
}
// Permutation key of node x.  A padding node gets the largest key.
__device__ __forceinline__ uint64_t perm_key(const SegKey& k, int64_t x) {
  const int64_t l = x - k.off;
  return l < k.n ? node_key(k.seed, static_cast<uint32_t>(l), k.g) : ~0ull;
}
// The graph that bucket b belongs to.
__device__ __forceinline__ int seg_of_bucket(const KeySrc& ks, int nseg, int64_t b) {
  int lo = 0, hi = nseg;
  while (hi - lo > 1) {
    const int mid = (lo + hi) >> 1;
    if (__ldg(&ks.segs[mid].bucket_base) <= b) lo = mid; else hi = mid;
  }
  return lo;
}

// ------------------------------------------- relaxed global trade (no sort)
//
// Def. "Relaxed global trade" with a linear congruential map
// h(x) = (a x + b) mod p, p the smallest prime >= n: the nodes in order of
// h(x).  The image of [n] is Z_p minus the p - n values h takes on [n, p)
// (the gaps; p - n is below a few hundred for any n < 2^31), so node x sits
// at position h(x) - #{gaps below h(x)}, with no sort.  (a, b) come from
// Philox4x32-10 on counter (0, 0, g, 4): a = 1 + (r0r1 mod (p-1)),
// b = r2r3 mod p.

__device__ __forceinline__ uint64_t mulmod(uint64_t x, uint64_t y, uint64_t p) { return (x * y) % p; }

// One CTA: (a, b) of the step, the gap values h(x), n <= x < p, sorted into gaps[1..]
// (gaps[0] = their count).
__global__ void k_lcg_gaps(int64_t n, uint64_t p, KeySrc ks, uint64_t* __restrict__ ab, int64_t* __restrict__ gaps) {
  __shared__ int64_t sg[kMaxLcgGaps];
  const uint64_t seed = ks.segs ? ks.segs[0].seed : ks.s0.seed;
  const uint32_t g = ks.use_abs ? ks.g_abs : (ks.segs ? ks.segs[0].g : ks.s0.g) + ks.dg;
  const Philox4 r = philox4x32_10(0u, 0u, g, 4u, seed);
  const uint64_t a = 1 + (((static_cast<uint64_t>(r.w0) << 32) | r.w1) % (p - 1));
  const uint64_t b = ((static_cast<uint64_t>(r.w2) << 32) | r.w3) % p;
  const int ng = static_cast<int>(p - static_cast<uint64_t>(n));
  int P = 1;
  while (P < ng) P <<= 1;
  for (int i = threadIdx.x; i < P; i += blockDim.x)
    sg[i] = i < ng ? static_cast<int64_t>((mulmod(a, static_cast<uint64_t>(n + i), p) + b) % p) : INT64_MAX;
  __syncthreads();
  for (int k = 2; k <= P; k <<= 1)
    for (int j = k >> 1; j > 0; j >>= 1) {
      for (int i = threadIdx.x; i < P; i += blockDim.x) {
        const int l = i ^ j;
        if (l > i) {
          const int64_t x = sg[i], y = sg[l];
          if ((x > y) == ((i & k) == 0)) { sg[i] = y; sg[l] = x; }
        }
      }
      __syncthreads();
    }
  for (int i = threadIdx.x; i < ng; i += blockDim.x) gaps[1 + i] = sg[i];
  if (threadIdx.x == 0) {
    gaps[0] = ng;
    ab[0] = a;
    ab[1] = b;
  }
}

// Node x goes to position h(x) - #{gaps < h(x)}.
__global__ void k_lcg_positions(int64_t n, uint64_t p, const uint64_t* __restrict__ ab,
                                const int64_t* __restrict__ gaps, int32_t* __restrict__ order,
                                int32_t* __restrict__ pos) {
  __shared__ int64_t sg[kMaxLcgGaps];
  const int ng = static_cast<int>(gaps[0]);
  for (int i = threadIdx.x; i < ng; i += blockDim.x) sg[i] = gaps[1 + i];
  __syncthreads();
  const uint64_t a = ab[0], b = ab[1];
  for (int64_t x = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; x < n; x += int64_t(gridDim.x) * blockDim.x) {
    const int64_t y = static_cast<int64_t>((mulmod(a, static_cast<uint64_t>(x), p) + b) % p);
    int lo = 0, hi = ng;   // gaps below y
    while (lo < hi) {
      const int mid = (lo + hi) >> 1;
      if (sg[mid] < y) lo = mid + 1; else hi = mid;
    }
    const int64_t q = y - lo;
    order[q] = static_cast<int32_t>(x);
    if (pos) pos[x] = static_cast<int32_t>(q);
  }
}

__device__ __forceinline__ bool pair_less(uint64_t ka, int32_t ia, uint64_t kb, int32_t ib) {
  return ka < kb || (ka == kb && ia < ib);
}

// What a bucket's sort writes: order and (may be null) positions, row offsets.
struct PermOut {
  int32_t* order;
  int32_t* pos;
  int64_t* rp;
  const int32_t* deg;   // degree by node id (for rp)
  int32_t* chunk_row;   // (may be null) the row of every kRowChunk-th entry
};
// Row p holds entries [e, e + d).
__device__ __forceinline__ void put_row(const PermOut& out, int64_t p, int64_t e, int64_t d) {
  out.rp[p] = e;
  if (!out.chunk_row) return;
  for (int64_t ch = (e + kRowChunk - 1) / kRowChunk; ch * kRowChunk < e + d; ++ch)
    out.chunk_row[ch] = static_cast<int32_t>(p);
}
// The end of the offsets, by one thread.
__device__ __forceinline__ void put_rows_end(const PermOut& out, int64_t n, int64_t nnz) {
  out.rp[n] = nnz;
  if (out.chunk_row) out.chunk_row[(nnz + kRowChunk - 1) / kRowChunk] = static_cast<int32_t>(n - 1);
}

constexpr int kSubBits = 10;
constexpr int kSubBins = 1 << kSubBits;
// dynamic shared memory for `cap` keys: keys, ids, degrees by rank, bin
// starts (+1), bin cursors, and each bin slot's element
size_t bucket_smem_bytes(int cap) {
  return static_cast<size_t>(cap) * (sizeof(uint64_t) + 2 * sizeof(int32_t) + sizeof(uint16_t)) +
         (2 * kSubBins + 2) * sizeof(int32_t);
}
struct BucketWs {
  uint64_t* key;
  int32_t* id;
  int32_t* sdeg;
  int32_t* bstart;   // kSubBins + 1
  int32_t* bcur;     // kSubBins
  uint16_t* slot;
};
__device__ __forceinline__ BucketWs bucket_ws(void* base, int cap) {
  BucketWs w;
  w.key = static_cast<uint64_t*>(base);
  w.id = reinterpret_cast<int32_t*>(w.key + cap);
  w.sdeg = w.id + cap;
  w.bstart = w.sdeg + cap;
  w.bcur = w.bstart + kSubBins + 1;
  w.slot = reinterpret_cast<uint16_t*>(w.bcur + kSubBins + 1);
  return w;
}

// Exclusive prefix sum over the CTA of NT threads, and the total.
template <int NT>
__device__ __forceinline__ int64_t cta_scan(int64_t v, int64_t* wsum, int64_t* total) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  int64_t incl = v;
#pragma unroll
  for (int off = 1; off < 32; off <<= 1) {
    const int64_t y = __shfl_up_sync(kFull, incl, off);
    if (lane >= off) incl += y;
  }
  if (lane == 31) wsum[warp] = incl;
  __syncthreads();
  int64_t before = 0, all = 0;
#pragma unroll
  for (int w = 0; w < NT / 32; ++w) {
    if (w < warp) before += wsum[w];
    all += wsum[w];
  }
  __syncthreads();
  *total = all;
  return incl - v + before;
}

// The s keys of a bucket in shared memory, to positions p0.. and entries
// e0..: a counting sort on the kSubBits bits below the highest bit where they
// differ (keys agree above it, so the digit orders them).
template <int NT>
__device__ void sort_bucket(const BucketWs& w, int s, int64_t p0, int64_t e0, const PermOut& out) {
  __shared__ unsigned long long s_or, s_and;
  __shared__ int64_t wsum[NT / 32];
  constexpr int kPer = kSubBins / NT;   // bins per thread in the scan
  const int lane = threadIdx.x & 31;
  if (threadIdx.x == 0) {
    s_or = 0ull;
    s_and = ~0ull;
  }
  for (int i = threadIdx.x; i < kSubBins; i += NT) w.bcur[i] = 0;
  __syncthreads();
  unsigned long long lor = 0ull, land = ~0ull;
  for (int i = threadIdx.x; i < s; i += NT) {
    lor |= w.key[i];
    land &= w.key[i];
  }
#pragma unroll
  for (int off = 16; off; off >>= 1) {
    lor |= __shfl_xor_sync(kFull, lor, off);
    land &= __shfl_xor_sync(kFull, land, off);
  }
  if (lane == 0) {
    atomicOr(&s_or, lor);
    atomicAnd(&s_and, land);
  }
  __syncthreads();
  const uint64_t diff = s_or ^ s_and;            // the bits where the bucket's keys differ
  const int top = diff ? 63 - __clzll(static_cast<long long>(diff)) : 0;
  const int sh = top + 1 > kSubBits ? top + 1 - kSubBits : 0;
  for (int i = threadIdx.x; i < s; i += NT)
    atomicAdd(&w.bcur[static_cast<int>(w.key[i] >> sh) & (kSubBins - 1)], 1);
  __syncthreads();
  // exclusive scan of the bin counts: kPer consecutive bins per thread
  int local = 0;
#pragma unroll
  for (int q = 0; q < kPer; ++q) local += w.bcur[threadIdx.x * kPer + q];
  int64_t all;
  int run = static_cast<int>(cta_scan<NT>(local, wsum, &all));
#pragma unroll
  for (int q = 0; q < kPer; ++q) {
    const int bi = threadIdx.x * kPer + q;
    const int c = w.bcur[bi];
    w.bstart[bi] = run;
    w.bcur[bi] = run;   // now the bin's cursor
    run += c;
  }
  if (threadIdx.x == 0) w.bstart[kSubBins] = s;
  __syncthreads();
  for (int i = threadIdx.x; i < s; i += NT)
    w.slot[atomicAdd(&w.bcur[static_cast<int>(w.key[i] >> sh) & (kSubBins - 1)], 1)] = static_cast<uint16_t>(i);
  __syncthreads();
  // rank within the bin: the bin's start plus the smaller (key, id) in it
  for (int i = threadIdx.x; i < s; i += NT) {
    const uint64_t ki = w.key[i];
    const int32_t ii = w.id[i];
    const int d = static_cast<int>(ki >> sh) & (kSubBins - 1);
    const int st = w.bstart[d], en = w.bstart[d + 1];
    int r = st;
    for (int q = st; q < en; ++q) {
      const int j = w.slot[q];
      r += (j != i && pair_less(w.key[j], w.id[j], ki, ii)) ? 1 : 0;
    }
    out.order[p0 + r] = ii;
    if (out.pos) out.pos[ii] = static_cast<int32_t>(p0 + r);
    if (out.rp) w.sdeg[r] = out.deg[ii];
  }
  __syncthreads();
  if (!out.rp) return;
  for (int base = 0; base < s; base += NT) {
    const int r = base + static_cast<int>(threadIdx.x);
    int64_t tot;
    const int64_t d = r < s ? w.sdeg[r] : 0;
    const int64_t x = cta_scan<NT>(d, wsum, &tot);
    if (r < s) put_row(out, p0 + r, e0 + x, d);
    e0 += tot;
  }
}

// A bucket that does not fit: get(i, &key, &id) enumerates candidates
// i < count and says which belong to the bucket; each is ranked against all
// others (keys computed anew each time).
template <int NT, class Get>
__device__ void rank_bucket(int64_t count, Get get, int64_t s, int64_t p0, int64_t e0, const PermOut& out) {
  __shared__ int64_t wsum[NT / 32];
  for (int64_t i = threadIdx.x; i < count; i += NT) {
    uint64_t ki, kj;
    int32_t ii, ij;
    if (!get(i, &ki, &ii)) continue;
    int64_t r = 0;
    for (int64_t j = 0; j < count; ++j) r += get(j, &kj, &ij) && pair_less(kj, ij, ki, ii) ? 1 : 0;
    out.order[p0 + r] = ii;
    if (out.pos) out.pos[ii] = static_cast<int32_t>(p0 + r);
    if (out.rp) out.rp[p0 + r] = out.deg[ii];   // replaced by its offset below
  }
  __syncthreads();
  if (!out.rp) return;
  for (int64_t base = 0; base < s; base += NT) {
    const int64_t r = base + threadIdx.x;
    int64_t tot;
    const int64_t d = r < s ? out.rp[p0 + r] : 0;
    const int64_t x = cta_scan<NT>(d, wsum, &tot);
    if (r < s) put_row(out, p0 + r, e0 + x, d);
    e0 += tot;
  }
}

// A bucket's word: nodes in it (bits 33..63) and their degrees summed (bits
// 0..32); n < 2^31 and row_ptr[n] < 2^33, so prefix sums over the words of a
// handle keep both fields.
constexpr int kCountShift = 33;
constexpr uint64_t kDegMask = (uint64_t(1) << kCountShift) - 1;

// Small handles: CTA b computes every key of its bucket's graph.  It costs
// span x buckets keys per graph; the launch and the memory round trip it saves
// cost more up to kRescanWork keys.  The latency of a thread's keys bounds it,
// so 1024 threads share them, degrees are loaded whether needed or not, and
// the next keys do not wait for the last ones (a permutation of 4096 nodes on
// its own: 12.3 us per call with 256 threads, 10.2 so).
constexpr int kRescanThreads = 1024;
__device__ void perm_rescan(int64_t n, int nseg, const KeySrc& ks, int nb, int cap, const PermOut& out,
                            const int64_t* rp_id, int64_t nnz, const ClassArgs& ca) {
  extern __shared__ uint64_t shk[];
  __shared__ int cnt;
  __shared__ int64_t wsum[kRescanThreads / 32];
  if (static_cast<int>(blockIdx.x) >= nb) {
    classify<kRescanThreads>(ca, blockIdx.x - nb, gridDim.x - nb);
    return;
  }
  const int64_t b = blockIdx.x;
  const SegKey k = seg_key(ks, nseg > 1 ? seg_of_bucket(ks, nseg, b) : 0);
  const uint32_t mine = static_cast<uint32_t>(b - k.base);
  const BucketWs w = bucket_ws(shk, cap);
  if (threadIdx.x == 0) cnt = 0;
  if (b == 0 && threadIdx.x == 0 && out.rp) put_rows_end(out, n, nnz);
  __syncthreads();
  const int64_t first_entry = out.rp ? rp_id[k.off] : 0;
  int64_t lower = 0, lower_deg = 0;
#pragma unroll 4
  for (int64_t x = k.off + threadIdx.x; x < k.off + k.span; x += kRescanThreads) {
    const int32_t d = out.rp ? out.deg[x] : 0;
    const uint64_t key = perm_key(k, x);
    const uint32_t bk = bucket_of(key, k.B);
    lower += bk < mine;
    lower_deg += bk < mine ? d : 0;
    if (bk == mine) {
      const int q = atomicAdd(&cnt, 1);
      if (q < cap) {
        w.key[q] = key;
        w.id[q] = static_cast<int32_t>(x);
      }
    }
  }
  // both sums in one scan: nodes below 2^31, entries below 2^33
  int64_t both;
  cta_scan<kRescanThreads>(static_cast<int64_t>((static_cast<uint64_t>(lower) << kCountShift) + static_cast<uint64_t>(lower_deg)),
                           wsum, &both);
  const int s = cnt;
  const int64_t p0 = k.off + static_cast<int64_t>(static_cast<uint64_t>(both) >> kCountShift);
  const int64_t e0 = first_entry + static_cast<int64_t>(static_cast<uint64_t>(both) & kDegMask);
  if (s <= cap) {
    sort_bucket<kRescanThreads>(w, s, p0, e0, out);
  } else {
    rank_bucket<kRescanThreads>(
        k.span,
        [&](int64_t i, uint64_t* key, int32_t* id) {
          *key = perm_key(k, k.off + i);
          *id = static_cast<int32_t>(k.off + i);
          return bucket_of(*key, k.B) == mine;
        },
        s, p0, e0, out);
  }
}
// beside: the kernel before it, the in-order pass, has started but may still
// run (it uses few SMs, and nothing that this kernel writes); the kernel after
// has to find both complete, so the wait comes last.
__global__ void __launch_bounds__(kRescanThreads) k_perm_rescan(int64_t n, int nseg, KeySrc ks, int nb, int cap,
                                                               PermOut out, const int64_t* rp_id,
                                                               int64_t nnz, ClassArgs ca, bool beside) {
  if (!beside) after_previous();
  before_next();
  perm_rescan(n, nseg, ks, nb, cap, out, rp_id, nnz, ca);
  if (beside) after_previous();
}
// 2^21 keys are 64 buckets of a 2^15-node graph: 128 keys per thread.
constexpr int64_t kRescanWork = int64_t(1) << 21;
constexpr int64_t kRescanBuckets = 4096;   // CTAs

// Node ids into their buckets (beside: as k_perm_rescan); the last CTA to finish turns the bucket words
// into their exclusive prefix sums and clears them for the next call.
__global__ void __launch_bounds__(kPermThreads) k_perm_scatter(int64_t n, KeySrc ks, int nb,
                                                              const int32_t* deg, unsigned long long* words,
                                                              uint64_t* prefix, int* ticket, int32_t* bid,
                                                              ClassArgs ca, bool beside) {
  if (!beside) after_previous();
  before_next();
  __shared__ int64_t wsum[kPermThreads / 32];
  __shared__ int last;
  classify<kPermThreads>(ca, blockIdx.x, gridDim.x);
  SegKey k = seg_key(ks, 0);
  int cur = 0;
  for (int64_t x = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; x < n; x += int64_t(gridDim.x) * blockDim.x) {
    if (ks.seg_of) {
      const int i = __ldg(ks.seg_of + x);
      if (i != cur) k = seg_key(ks, cur = i);
    }
    const uint32_t lb = bucket_of(perm_key(k, x), k.B);
    const unsigned long long inc =
        (1ull << kCountShift) + (deg ? static_cast<unsigned long long>(__ldg(deg + x)) : 0ull);
    const int64_t q = static_cast<int64_t>(atomicAdd(words + k.base + lb, inc) >> kCountShift);
    if (q < k.cap) bid[k.slot_base + int64_t(lb) * k.cap + q] = static_cast<int32_t>(x);
  }
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) last = atomicAdd(ticket, 1) == static_cast<int>(gridDim.x) - 1;
  __syncthreads();
  if (!last) return;
  __threadfence();
  uint64_t run = 0;
  constexpr int kPer = 8;
  for (int64_t base = 0; base < nb; base += kPermThreads * kPer) {
    const int64_t i0 = base + int64_t(threadIdx.x) * kPer;
    uint64_t v[kPer], sum = 0;
#pragma unroll
    for (int j = 0; j < kPer; ++j) {
      v[j] = i0 + j < nb ? __ldcg(words + i0 + j) : 0ull;
      sum += v[j];
    }
    int64_t tot;
    uint64_t p = run + static_cast<uint64_t>(cta_scan<kPermThreads>(static_cast<int64_t>(sum), wsum, &tot));
#pragma unroll
    for (int j = 0; j < kPer; ++j)
      if (i0 + j < nb) {
        prefix[i0 + j] = p;
        words[i0 + j] = 0ull;
        p += v[j];
      }
    run += static_cast<uint64_t>(tot);
  }
  if (threadIdx.x == 0) {
    prefix[nb] = run;
    *ticket = 0;
  }
  if (beside) after_previous();   // (the other CTAs need not stay)
}

__global__ void __launch_bounds__(kPermThreads) k_bucket_sort(int64_t n, int nseg, KeySrc ks, int nb, int cap,
                                                             const uint64_t* prefix, const int32_t* bid,
                                                             PermOut out, int64_t nnz, ClassArgs ca, bool beside) {
  if (!beside) after_previous();
  before_next();
  extern __shared__ uint64_t shk[];
  classify<kPermThreads>(ca, blockIdx.x, gridDim.x);
  const BucketWs w = bucket_ws(shk, cap);
  if (blockIdx.x == 0 && threadIdx.x == 0 && out.rp) put_rows_end(out, n, nnz);
  for (int64_t b = blockIdx.x; b < nb; b += gridDim.x) {
    const SegKey k = seg_key(ks, nseg > 1 ? seg_of_bucket(ks, nseg, b) : 0);
    const uint64_t p = prefix[b];
    const int64_t p0 = static_cast<int64_t>(p >> kCountShift), e0 = static_cast<int64_t>(p & kDegMask);
    const int64_t s = static_cast<int64_t>(prefix[b + 1] >> kCountShift) - p0;
    const uint32_t mine = static_cast<uint32_t>(b - k.base);
    const int32_t* ids = bid + k.slot_base + int64_t(mine) * k.cap;
    if (s <= cap && s <= k.cap) {
      for (int i = threadIdx.x; i < s; i += kPermThreads) {
        const int32_t x = ids[i];
        w.id[i] = x;
        w.key[i] = perm_key(k, x);
      }
      __syncthreads();
      sort_bucket<kPermThreads>(w, static_cast<int>(s), p0, e0, out);
    } else if (s <= k.cap) {   // above the shared-memory cap
      rank_bucket<kPermThreads>(
          s,
          [&](int64_t i, uint64_t* key, int32_t* id) {
            *id = ids[i];
            *key = perm_key(k, *id);
            return true;
          },
          s, p0, e0, out);
    } else {                   // the bucket's space did not hold all of it
      rank_bucket<kPermThreads>(
          k.span,
          [&](int64_t i, uint64_t* key, int32_t* id) {
            *key = perm_key(k, k.off + i);
            *id = static_cast<int32_t>(k.off + i);
            return bucket_of(*key, k.B) == mine;
          },
          s, p0, e0, out);
    }
    __syncthreads();
  }
  if (beside && blockIdx.x == 0) after_previous();
}

// Trades of the current step by size class, on its own (relaxed permutations).
__global__ void __launch_bounds__(kPermThreads) k_classify(ClassArgs ca) {
  classify<kPermThreads>(ca, blockIdx.x, gridDim.x);
}

__global__ void k_order_degrees(int64_t n, const int32_t* __restrict__ order, const int32_t* __restrict__ deg_id,
                                int32_t* __restrict__ out) {
  for (int64_t p = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; p < n; p += int64_t(gridDim.x) * blockDim.x)
    out[p] = deg_id[order[p]];
}

// The chunk rows of given offsets (see PermOut).
__global__ void k_chunk_rows(int64_t n, const int64_t* __restrict__ rp, int32_t* __restrict__ chunk_row) {
  for (int64_t p = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; p < n; p += int64_t(gridDim.x) * blockDim.x) {
    for (int64_t ch = (rp[p] + kRowChunk - 1) / kRowChunk; ch * kRowChunk < rp[p + 1]; ++ch)
      chunk_row[ch] = static_cast<int32_t>(p);
    if (p == n - 1) chunk_row[(rp[n] + kRowChunk - 1) / kRowChunk] = static_cast<int32_t>(p);
  }
}

struct PermWs {
  unsigned long long* words;   // nb, zero between calls
  int* ticket;                 // zero between calls
  uint64_t* prefix;            // nb + 1
  int32_t* bid;                // bucket spaces
};

size_t align_up(size_t x) { return (x + 255) & ~size_t(255); }

PermWs carve(void* base, int64_t nb) {
  char* p = static_cast<char*>(base);
  PermWs w;
  w.words = reinterpret_cast<unsigned long long*>(p); p += align_up(sizeof(unsigned long long) * nb);
  w.ticket = reinterpret_cast<int*>(p); p += 256;
  w.prefix = reinterpret_cast<uint64_t*>(p); p += align_up(sizeof(uint64_t) * (nb + 1));
  w.bid = reinterpret_cast<int32_t*>(p);
  return w;
}
size_t zero_bytes(int64_t nb) { return align_up(sizeof(unsigned long long) * nb) + 256; }

unsigned grid_for(int64_t work, int threads, int num_sms) {
  const int64_t want = (work + threads - 1) / threads;
  const int64_t cap = int64_t(num_sms) * 16;
  return static_cast<unsigned>(want < 1 ? 1 : (want < cap ? want : cap));
}

}  // namespace

bool perm_rescans(int64_t nbuckets, int64_t keys) { return nbuckets <= kRescanBuckets && keys <= kRescanWork; }

// Scratch of a handle: bucket words, prefixes, and `slots` ids of bucket space.
size_t perm_ws_bytes(int64_t nbuckets, int64_t slots) {
  return zero_bytes(nbuckets) + align_up(sizeof(uint64_t) * (nbuckets + 1)) + align_up(sizeof(int32_t) * slots);
}

// The bucket sort's shared memory for the largest "bucket_cap" (set once,
// outside any stream capture).
int init_perm_kernels(Graph* h) {
  CB_CUDA(h, cudaFuncSetAttribute(k_bucket_sort, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                  static_cast<int>(bucket_smem_bytes(kBucketCapMax))));
  CB_CUDA(h, cudaFuncSetAttribute(k_perm_rescan, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                  static_cast<int>(bucket_smem_bytes(kBucketCapMax))));
  return CB_OK;
}
size_t perm_zero_bytes(int64_t nbuckets) { return zero_bytes(nbuckets); }

namespace {
// Keys a rescan of every bucket would compute.
int64_t rescan_work(const Graph* h) {
  int64_t w = 0;
  for (int i = 0; i < h->nseg && w <= kRescanWork; ++i) w += h->hsegs[i].span << h->hsegs[i].B;
  return w;
}
int bucket_cap_of(const Graph* h) {
  int64_t cap = 1;
  for (int i = 0; i < h->nseg; ++i) cap = std::max<int64_t>(cap, h->hsegs[i].cap);
  return static_cast<int>(std::min<int64_t>(cap, h->bucket_cap));
}
}  // namespace

int compute_permutation(Graph* h, uint32_t dg, int64_t g_abs, int32_t* order_out, int32_t* pos_out, int64_t* rp_out,
                        const ClassArgs* classes, PermPart part) {
  const int64_t n = h->n;
  if (n == 0) return CB_OK;
  cudaStream_t s = h->stream;
  KeySrc ks{};
  ks.segs = h->segs;
  ks.dg = dg;
  ks.use_abs = g_abs >= 0;
  ks.g_abs = static_cast<uint32_t>(g_abs < 0 ? 0 : g_abs);
  ClassArgs ca{};
  if (classes) ca = *classes;
  const bool beside = part != PermPart::kWhole;
  const int64_t chunks = class_chunks(ca.ntasks, kPermThreads);
  if (h->relaxed) {
    if (ca.ntasks) {
      k_classify<<<static_cast<unsigned>(std::min<int64_t>(chunks, int64_t(h->num_sms) * 8)), kPermThreads, 0, s>>>(ca);
      CB_CUDA(h, cudaGetLastError());
      ++h->launches;
    }
    k_lcg_gaps<<<1, 256, 0, s>>>(n, h->lcg_p, ks, h->lcg_ab, h->lcg_gaps);
    CB_CUDA(h, cudaGetLastError());
    k_lcg_positions<<<grid_for(n, kPermThreads, h->num_sms), kPermThreads, 0, s>>>(n, h->lcg_p, h->lcg_ab, h->lcg_gaps,
                                                                                  order_out, pos_out);
    CB_CUDA(h, cudaGetLastError());
    h->launches += 2;
    if (rp_out) {
      int32_t* deg = reinterpret_cast<int32_t*>(h->thr_key);   // 8 bytes per trade, free until the first pass
      k_order_degrees<<<grid_for(n, kPermThreads, h->num_sms), kPermThreads, 0, s>>>(n, order_out, h->deg_id, deg);
      CB_CUDA(h, cudaGetLastError());
      ++h->launches;
      CB_CUDA(h, exclusive_scan_i32(deg, rp_out, n, h->scan_ws, s, &h->launches));
      k_chunk_rows<<<grid_for(n, kPermThreads, h->num_sms), kPermThreads, 0, s>>>(n, rp_out, h->chunk_row);
      CB_CUDA(h, cudaGetLastError());
      ++h->launches;
    }
    return CB_OK;
  }
  ks.seg_of = h->seg_of;
  const int64_t nb = h->nbuckets;
  const int cap = bucket_cap_of(h);
  const PermOut out{order_out, pos_out, rp_out, h->deg_id, !rp_out ? nullptr : beside ? h->chunk_row2 : h->chunk_row};
  if (perm_rescans(nb, rescan_work(h))) {
    if (part == PermPart::kScatterAhead) return CB_OK;
    const unsigned grid = static_cast<unsigned>(
        nb + std::min<int64_t>(class_chunks(ca.ntasks, kRescanThreads), int64_t(h->num_sms) * 2));
    CB_CUDA(h, launch(beside || small_handle(h), k_perm_rescan, grid, kRescanThreads, bucket_smem_bytes(cap), s, n, h->nseg,
                      ks, static_cast<int>(nb), cap, out, h->rp_id, h->nnz, ca, beside));
    ++h->launches;
    return CB_OK;
  }
  const PermWs w = carve(h->sort_ws, nb);
  const ClassArgs none{};
  if (part != PermPart::kRestAhead) {
    CB_CUDA(h, launch(beside || small_handle(h), k_perm_scatter, grid_for(n, kPermThreads, h->num_sms), kPermThreads, 0, s,
                      n, ks, static_cast<int>(nb), rp_out ? h->deg_id : nullptr, w.words, w.prefix, w.ticket, w.bid, ca,
                      beside));
    ++h->launches;
  }
  if (part != PermPart::kScatterAhead) {
    const unsigned sgrid = static_cast<unsigned>(nb < h->num_sms * 8 ? nb : h->num_sms * 8);
    CB_CUDA(h, launch(beside || small_handle(h), k_bucket_sort, sgrid, kPermThreads, bucket_smem_bytes(cap), s, n, h->nseg,
                      ks, static_cast<int>(nb), cap, w.prefix, w.bid, out, h->nnz, beside ? ca : none, beside));
    ++h->launches;
  }
  return CB_OK;
}

}  // namespace cb

// ---------------------------------------------------------------------------
// The permutation without any allocation: same key sort, with its scratch in
// a static device array instead of memory owned by a handle.  For callers
// that may not allocate device memory themselves -- for example code running
// under a host framework that owns every device allocation, or a latency-
// critical loop where cudaMalloc could synchronise the device or fail.
namespace cb {
namespace {
constexpr int64_t kStaticPermMaxNodes = int64_t(1) << 20;   // largest n accepted
constexpr size_t kStaticPermBytes = size_t(13) << 20;       // >= the scratch of any n up to 2^20
constexpr int kStaticPermMaxDevices = 64;
std::mutex g_static_perm_mu;
void* g_static_perm_ptr[kStaticPermMaxDevices] = {};
}  // namespace
}  // namespace cb

// Scratch of cb_permutation_static, shared by every call on a device and held
// by every device that loads the library until the process exits.
static __device__ __align__(256) unsigned char g_static_perm_scratch[cb::kStaticPermBytes];

extern "C" int cb_permutation_static(int64_t n, uint64_t seed, uint64_t g, int32_t* order_out,
                                     void* cuda_stream) {
  using namespace cb;
  if (n < 0 || (n > 0 && !order_out)) return fail(nullptr, CB_EINVAL, "cb_permutation_static: bad n or order_out");
  if (n > kStaticPermMaxNodes)
    return fail(nullptr, CB_ESIZE, "cb_permutation_static: n exceeds the static scratch limit of 2^20 nodes");
  if (g >= 0xfffffffeull) return fail(nullptr, CB_ERANGE, "cb_permutation_static: step too large");
  const int B = bucket_bits(n);
  const int nb = 1 << B;
  const int64_t space = bucket_space(n, B);
  if (perm_ws_bytes(nb, space * nb) > kStaticPermBytes)
    return fail(nullptr, CB_ECHECK, "cb_permutation_static: static scratch smaller than its limit needs");
  if (n == 0) return CB_OK;
  int dev = 0, num_sms = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return cuda_fail(nullptr, e, "cudaGetDevice");
  if (dev < 0 || dev >= kStaticPermMaxDevices) return fail(nullptr, CB_EINVAL, "cb_permutation_static: device index");
  void* base = nullptr;
  {
    // once per device, with that device current: the device address of the scratch
    std::lock_guard<std::mutex> lock(g_static_perm_mu);
    if (!g_static_perm_ptr[dev]) {
      void* p = nullptr;
      e = cudaGetSymbolAddress(&p, g_static_perm_scratch);
      if (e != cudaSuccess) return cuda_fail(nullptr, e, "cudaGetSymbolAddress");
      g_static_perm_ptr[dev] = p;
    }
    base = g_static_perm_ptr[dev];
  }
  e = cudaDeviceGetAttribute(&num_sms, cudaDevAttrMultiProcessorCount, dev);
  if (e != cudaSuccess) return cuda_fail(nullptr, e, "cudaDeviceGetAttribute");
  cudaStream_t s = static_cast<cudaStream_t>(cuda_stream);
  KeySrc ks{};
  ks.s0.seed = seed;
  ks.s0.n = n;
  ks.s0.span = n;
  ks.s0.B = B;
  ks.s0.cap = static_cast<int32_t>(space);
  ks.use_abs = 1;
  ks.g_abs = static_cast<uint32_t>(g);
  const PermOut out{order_out, nullptr, nullptr, nullptr, nullptr};
  // at most 2048 keys of a bucket in shared memory (45 KB: no attribute needed)
  const int cap = static_cast<int>(std::min<int64_t>(space, 2048));
  const ClassArgs none{};
  if (n * nb <= kRescanWork) {   // no scratch at all
    k_perm_rescan<<<nb, kRescanThreads, bucket_smem_bytes(cap), s>>>(n, 1, ks, nb, cap, out, nullptr, 0, none, false);
    if ((e = cudaGetLastError()) != cudaSuccess) return cuda_fail(nullptr, e, "k_perm_rescan");
    return CB_OK;
  }
  // the scratch keeps the previous call's contents: clear the bucket words
  const PermWs w = carve(base, nb);
  if ((e = cudaMemsetAsync(base, 0, zero_bytes(nb), s)) != cudaSuccess) return cuda_fail(nullptr, e, "cudaMemsetAsync");
  k_perm_scatter<<<grid_for(n, kPermThreads, num_sms), kPermThreads, 0, s>>>(n, ks, nb, nullptr, w.words, w.prefix,
                                                                            w.ticket, w.bid, none, false);
  if ((e = cudaGetLastError()) != cudaSuccess) return cuda_fail(nullptr, e, "k_perm_scatter");
  const unsigned sgrid = static_cast<unsigned>(nb < num_sms * 8 ? nb : num_sms * 8);
  k_bucket_sort<<<sgrid, kPermThreads, bucket_smem_bytes(cap), s>>>(n, 1, ks, nb, cap, w.prefix, w.bid, out, 0, none, false);
  if ((e = cudaGetLastError()) != cudaSuccess) return cuda_fail(nullptr, e, "k_bucket_sort");
  return CB_OK;
}

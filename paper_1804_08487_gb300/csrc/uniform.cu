// Uniform single trades (Simple Undirected Curveball, Section 3.2) on the
// device, and the successor lists Suc of a trade sequence (Section 4.1).
//
// The sequence runs as a dataflow in the manner of EM-CB / IM-CB (Sections
// 4.1-4.2) on node ids (a trade's keys are functions of ids); the input rows
// and the output are in the position space of the handle's current super step:
//   - Suc gives, for every (trade, endpoint), the endpoint's next trade, and
//     for every node its first trade.
//   - Every edge waits in an inbox of the next trade of either endpoint:
//     that trade is the only one that can change it.
//   - An inbox entry carries the neighbour and the neighbour's next trade.
//     Trade k's inbox for node x has deg(x) slots, reserved by one 64-bit
//     atomic per entry (both sides' counts packed).
//   - The reservation that fills the last slot queues the trade.
//   - Persistent CTAs take queued trades in queue order: trades of at most
//     128 (or 64) entries one per warp, larger ones on a team of three quarters
//     of the CTA's threads.  Each trade:
//       - gathers both inboxes, waiting (bounded) for entries still being
//         written;
//       - finds the common and disjoint neighbours through a hash of u's
//         neighbours;
//       - finds the threshold of sigma(D) by a radix select on D's keys;
//       - sends every resulting edge on.
//   - An edge whose endpoints both have no further trade goes to its rows of
//     the output.
// The critical path of the dataflow is a chain of dependent trades. So a
// trade's own latency counts: no sort, few barriers, and the atomics of a
// thread's messages in flight together.
// Every trade sees exactly the neighbourhoods it would see in index order:
// an edge {a, b} changes only in trades of a or b, and it reaches the first
// of those before anything else touches it.
#include <algorithm>
#include <cstring>

#include "cb_internal.cuh"
#include "philox.cuh"
#include "run_queues.cuh"
#include "team.cuh"

namespace cb {

struct UniBufs {
  int64_t cap_trades = 0;      // trades per chunk the buffers hold
  int64_t n = 0;
  int32_t* tp = nullptr;       // 2L: u_i (even) and v_i (odd)
  int32_t* dslot = nullptr;    // 2L: degree of each slot's node
  int64_t* ib = nullptr;       // 2L+1: first inbox entry of each slot
  int32_t* suc = nullptr;      // 2L: slot ids grouped by node, increasing
  int32_t* nxt = nullptr;      // 2L: next slot of the slot's node
  unsigned long long* fill = nullptr;   // L: inbox counts (side 0 low, side 1 high)
  int32_t* queue = nullptr;    // L: runnable trades; small ones from the front, big ones from the back
  int32_t* occ = nullptr;      // n: occurrences, then fill cursors
  int32_t* first = nullptr;    // n: first slot of the node at each position
  int64_t* sbeg = nullptr;     // n+1: Suc offsets
  int32_t* ocur = nullptr;     // n: output row cursors
  unsigned long long* ctr = nullptr;   // heads and tails of the two run queues, a cache line apart
  void* scan_ws = nullptr;
  int2* inbox = nullptr;
  int64_t inbox_cap = 0;
  char* gslice = nullptr;      // per-CTA work space for trades above the shared-memory cap
  int64_t slice_elems = 0;
  int ctas = 0;
  size_t bytes = 0, inbox_bytes = 0, slice_bytes = 0;
};

namespace {

// "Next trade" of a node is its slot there, 2 trade + side, so that a message
// knows its side without a look at the trade; kInf: no further trade.
constexpr int32_t kInf = 0x7fffffff;
__device__ __forceinline__ int32_t trade_of(int32_t slot) { return slot == kInf ? kInf : slot >> 1; }
// Executor CTAs of NT = 256, 512 or 1024 threads (option "uniform_threads"):
// three quarters of them are one team for large trades, the other warps take the small trades one each, and so do the
// team's warps once the large trades are all taken.  Every CTA serves both
// queues, so whichever CTAs are resident finish the sequence.  A larger team
// makes the hub trades on the critical chain shorter.
template <int NT>
__host__ __device__ constexpr int uni_team() { return NT / 4 * 3; }
template <int NT>
__host__ __device__ constexpr int uni_warps() { return NT / 128; }
template <int NT>
__host__ __device__ constexpr int uni_smem_elems() { return NT == 1024 ? 4096 : 2048; }   // trades up to this many entries in shared memory
// Small trades have at most kUniSmall entries (four per lane of a warp), in
// chunks of at most kUniFewMax trades half as many: there the chain of
// dependent trades bounds the time, and a team finishes a trade of 65 to 128
// entries sooner than a warp; in longer chunks the teams are too few for them.
// 64 against 128 entries: n=2^14 0.54 and 0.74 ms, 2^17 2.03 and 2.10, 2^20
// 11.0 and 10.2 (n/2 trades each).
constexpr int kUniSmall = 128;
constexpr int64_t kUniFewMax = 65536;
inline int uni_small(int64_t trades) { return trades <= kUniFewMax ? kUniSmall / 2 : kUniSmall; }
constexpr int64_t kUniChunkMin = 65536;

__device__ __forceinline__ void latch(int32_t* err, int32_t code) { atomicCAS(err, 0, code); }

__device__ __forceinline__ uint64_t globaltimer() {
  uint64_t t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

__device__ __forceinline__ int32_t ld_volatile_i32(const int32_t* p) {
  return *reinterpret_cast<const volatile int32_t*>(p);
}

__device__ __forceinline__ int2 ld_relaxed_v2(const int2* p) {
  int2 v;
  asm volatile("ld.relaxed.gpu.global.v2.s32 {%0, %1}, [%2];" : "=r"(v.x), "=r"(v.y) : "l"(p) : "memory");
  return v;
}

__device__ __forceinline__ void st_relaxed_v2(int2* p, int32_t x, int32_t y) {
  asm volatile("st.relaxed.gpu.global.v2.s32 [%0], {%1, %2};" ::"l"(p), "r"(x), "r"(y) : "memory");
}

__device__ __forceinline__ void st_relaxed_i32(int32_t* p, int32_t x) {
  asm volatile("st.relaxed.gpu.global.s32 [%0], %1;" ::"l"(p), "r"(x) : "memory");
}

__device__ __forceinline__ int32_t ld_relaxed_i32(const int32_t* p) {
  int32_t v;
  asm volatile("ld.relaxed.gpu.global.s32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}

// ------------------------------------------------------------- the sequence

// Pair of trade i on n >= 2 nodes: counter (i_lo, i_hi, 0, 5), multiply-high
// maps of words 0 and 1 (see cb_uniform.h).
__device__ __forceinline__ void uniform_pair(uint64_t seed, int64_t n, uint64_t i, int32_t* u, int32_t* v) {
  const Philox4 r = philox4x32_10(static_cast<uint32_t>(i), static_cast<uint32_t>(i >> 32), 0u, 5u, seed);
  const int64_t a = static_cast<int64_t>((static_cast<uint64_t>(r.w0) * static_cast<uint64_t>(n)) >> 32);
  const int64_t w = static_cast<int64_t>((static_cast<uint64_t>(r.w1) * static_cast<uint64_t>(n - 1)) >> 32);
  *u = static_cast<int32_t>(a);
  *v = static_cast<int32_t>(w + (w >= a));
}

// pairs of trades first..first+count-1; with the nodes' degrees, each slot's
// goes to dslot, its node's occurrences are counted and *big counts trades of
// more than small entries.
__global__ void k_uni_draw(int64_t count, uint64_t first, uint64_t seed, int64_t n, const int32_t* __restrict__ deg,
                           int32_t* __restrict__ out, int32_t* __restrict__ dslot,
                           int32_t* __restrict__ occ, int small, unsigned long long* __restrict__ big) {
  int large = 0;
  for (int64_t i = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; i < count; i += int64_t(gridDim.x) * blockDim.x) {
    int32_t u, v;
    uniform_pair(seed, n, first + static_cast<uint64_t>(i), &u, &v);
    out[2 * i] = u;
    out[2 * i + 1] = v;
    if (dslot) {
      const int32_t du = deg[u], dv = deg[v];
      dslot[2 * i] = du;
      dslot[2 * i + 1] = dv;
      large += int64_t(du) + dv > small;
      atomicAdd(&occ[u], 1);
      atomicAdd(&occ[v], 1);
    }
  }
  if (dslot) {
    large = __reduce_add_sync(kFull, large);
    if ((threadIdx.x & 31) == 0 && large) atomicAdd(big, static_cast<unsigned long long>(large));
  }
}

// occ[x] = number of slots naming x; pairs out of range or with equal nodes latch err.
__global__ void k_uni_count(int64_t count, int64_t n, const int32_t* __restrict__ tp, int32_t* __restrict__ occ,
                            int32_t* err) {
  for (int64_t i = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; i < count; i += int64_t(gridDim.x) * blockDim.x) {
    const int32_t a = tp[2 * i], b = tp[2 * i + 1];
    if (a < 0 || b < 0 || a >= n || b >= n || a == b) {
      latch(err, kErrValidate);
      continue;
    }
    atomicAdd(&occ[a], 1);
    atomicAdd(&occ[b], 1);
  }
}

// suc[sbeg[x] + k] = slot ids of x (unordered; cursors start at 0)
__global__ void k_uni_fill(int64_t slots, const int32_t* __restrict__ tp, const int64_t* __restrict__ sbeg,
                           int32_t* __restrict__ cursor, int32_t* __restrict__ suc) {
  for (int64_t j = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; j < slots; j += int64_t(gridDim.x) * blockDim.x) {
    const int32_t x = tp[j];
    const int32_t k = atomicAdd(&cursor[x], 1);
    suc[sbeg[x] + k] = static_cast<int32_t>(j);
  }
}

// Each node's slot list in increasing order (a node is in a trade at most
// once, so slot order is trade order); with nxt, every slot's next slot and
// every node's first one at its position.
__global__ void k_uni_sort(int64_t n, const int64_t* __restrict__ sbeg, int32_t* __restrict__ suc,
                           int32_t* __restrict__ nxt, const int32_t* __restrict__ pos, int32_t* __restrict__ first) {
  for (int64_t x = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; x < n; x += int64_t(gridDim.x) * blockDim.x) {
    const int64_t b = sbeg[x], e = sbeg[x + 1];
    for (int64_t i = b + 1; i < e; ++i) {   // lists are short: Poisson(2L/n) long
      const int32_t key = suc[i];
      int64_t j = i - 1;
      while (j >= b && suc[j] > key) {
        suc[j + 1] = suc[j];
        --j;
      }
      suc[j + 1] = key;
    }
    if (nxt) {
      first[pos[x]] = b < e ? suc[b] : kInf;
      for (int64_t i = b; i < e; ++i) nxt[suc[i]] = (i + 1 < e) ? suc[i + 1] : kInf;
    }
  }
}

__global__ void k_uni_trade_index(int64_t slots, const int32_t* __restrict__ suc, int32_t* __restrict__ out) {
  for (int64_t j = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; j < slots; j += int64_t(gridDim.x) * blockDim.x)
    out[j] = suc[j] >> 1;
}

// ------------------------------------------------------------- the dataflow

struct UniCtx {
  int64_t L;                 // trades in this chunk
  uint64_t first;            // global index of the chunk's first trade
  uint64_t seed;
  const int64_t* rp;         // position-space row offsets (degrees never change)
  const int32_t* order;      // node id at each position
  const int32_t* pos;        // position of each node id
  const int32_t* tp;
  const int32_t* dslot;
  const int32_t* nxt;
  const int64_t* ib;
  const int32_t* first_slot;   // of the node at each position
  int2* inbox;
  unsigned long long* fill;
  int32_t* queue;
  unsigned long long* ctr;
  int32_t* ocur;
  int32_t* col_out;
  int32_t* err;
  char* gslice;
  int64_t slice_elems;
  unsigned long long* swaps;   // (performed, possible) swap counts, or null
  uint64_t wait_ns;            // longest single wait (run queue, inbox entry)
  int small;                   // entries of the largest small trade, at most kUniSmall
  int64_t hold_trade;          // test hook: messages to this trade of the chunk are dropped (-1: none)
};

// The two run queues (run_queues.cuh): a ticket (kHead) takes the queue's next
// place, a push (kTail) fills the next place; the counters sit on different
// cache lines.  Every trade is queued exactly once and kBig says how many are
// large, so every ticket below a queue's length ends; a push past it latches
// the error and touches no place.
constexpr int kHead = 0, kTail = 16, kQueueCtr = 32, kBig = 64, kCtrWords = 80;

__device__ __forceinline__ RunQueues queues(const UniCtx& c) { return {c.L, static_cast<int64_t>(c.ctr[kBig])}; }

__device__ __forceinline__ void push(const UniCtx& c, int64_t k, int64_t entries) {
  const int big = entries > c.small;
  const RunQueues rq = queues(c);
  const unsigned long long q = atomicAdd(&c.ctr[kQueueCtr * big + kTail], 1ull);
  if (!rq.holds(big, q)) {
    latch(c.err, kErrUniform);
    return;
  }
  st_relaxed_i32(c.queue + rq.place(big, q), static_cast<int32_t>(k));
}

// The next queued trade, or -1 when every place of the queue is taken or a
// wait gave up.
__device__ int64_t take_ticket(const UniCtx& c, int big, const RunQueues& rq) {
  const unsigned long long q = atomicAdd(&c.ctr[kQueueCtr * big + kHead], 1ull);
  if (!rq.holds(big, q)) return -1;
  const int32_t* place = c.queue + rq.place(big, q);
  int32_t t = ld_relaxed_i32(place);
  if (t < 0) {
    const uint64_t t0 = globaltimer();
    for (;;) {
      __nanosleep(200);
      t = ld_relaxed_i32(place);
      if (t >= 0) break;
      if (ld_volatile_i32(c.err) != 0) return -1;
      if (globaltimer() - t0 > c.wait_ns) {
        latch(c.err, kErrUniformWait);
        return -1;
      }
    }
  }
  return t;
}

// One message: the edge {a, b} with a's next slot ta and b's next slot tb, to
// the earlier of the two trades (both inboxes when they are the same trade),
// or out.  reserve() takes the places (one atomic per message) and loads what
// deliver(), which writes them, needs of the destination.
struct Msg {
  int32_t a, ta, b, tb, d;
  unsigned long long old;   // previous inbox counts of trade d, or the two row cursors
  int64_t ib;
  int2 deg;                 // the destination's degrees, or the positions of a and b
};

__device__ __forceinline__ unsigned long long msg_inc(const Msg& m) {
  unsigned long long inc = 0;
  if (trade_of(m.ta) == m.d) inc += (m.ta & 1) ? (1ull << 32) : 1ull;
  if (trade_of(m.tb) == m.d) inc += (m.tb & 1) ? (1ull << 32) : 1ull;
  return inc;
}

__device__ __forceinline__ void reserve(const UniCtx& c, Msg& m) {
  m.d = min(trade_of(m.ta), trade_of(m.tb));
  if (m.d == kInf) {
    m.deg = make_int2(c.pos[m.a], c.pos[m.b]);
    const uint32_t sa = static_cast<uint32_t>(atomicAdd(&c.ocur[m.deg.x], 1));
    const uint32_t sb = static_cast<uint32_t>(atomicAdd(&c.ocur[m.deg.y], 1));
    m.old = (static_cast<unsigned long long>(sb) << 32) | sa;
    return;
  }
  m.old = atomicAdd(&c.fill[m.d], msg_inc(m));
  m.ib = c.ib[2 * int64_t(m.d)];
  m.deg = reinterpret_cast<const int2*>(c.dslot)[m.d];
}

// places s0, s1: the entry's place on its side of trade d
__device__ __forceinline__ void put_entry(const UniCtx& c, const Msg& m, int side, int32_t other, int32_t other_tau) {
  const uint32_t place = static_cast<uint32_t>(side ? m.old >> 32 : m.old);
  if (place >= static_cast<uint32_t>(side ? m.deg.y : m.deg.x)) {
    latch(c.err, kErrUniform);
    return;
  }
  st_relaxed_v2(c.inbox + m.ib + (side ? m.deg.x : 0) + place, other, other_tau);
}

__device__ __forceinline__ void deliver(const UniCtx& c, const Msg& m) {
  if (m.d == kInf) {
    const int32_t pa = m.deg.x, pb = m.deg.y;
    const int64_t ba = c.rp[pa], bb = c.rp[pb];
    const uint32_t sa = static_cast<uint32_t>(m.old), sb = static_cast<uint32_t>(m.old >> 32);
    if (sa < c.rp[pa + 1] - ba) c.col_out[ba + sa] = pb;
    else latch(c.err, kErrRowLength);
    if (sb < c.rp[pb + 1] - bb) c.col_out[bb + sb] = pa;
    else latch(c.err, kErrRowLength);
    return;
  }
  if (trade_of(m.ta) == m.d) put_entry(c, m, m.ta & 1, m.b, m.tb);
  if (trade_of(m.tb) == m.d) put_entry(c, m, m.tb & 1, m.a, m.ta);
  const unsigned long long full =
      (static_cast<unsigned long long>(static_cast<uint32_t>(m.deg.y)) << 32) | static_cast<uint32_t>(m.deg.x);
  if (m.old + msg_inc(m) == full) push(c, m.d, int64_t(m.deg.x) + m.deg.y);
}

// Every edge of the input to the first trade of either endpoint; trades with
// no entries to wait for are queued here.  The edges of a row that go to the
// row's own first trade take their places with one atomic per 32 of them.
// Scattered L2 accesses bound it, about six per edge (24 million edges, n=2^20:
// 1.05 ms).
__global__ void k_uni_route(UniCtx c, int64_t n, const int32_t* __restrict__ col) {
  const int lane = threadIdx.x & 31;
  const int64_t gw = (blockIdx.x * int64_t(blockDim.x) + threadIdx.x) >> 5;
  const int64_t nw = int64_t(gridDim.x) * (blockDim.x >> 5);
  for (int64_t a = gw; a < n; a += nw) {
    const int64_t b0 = c.rp[a], b1 = c.rp[a + 1];
    if (b0 == b1) continue;
    const int32_t ta = c.first_slot[a], da = trade_of(ta), ida = c.order[a];
    int64_t ib = 0;
    int2 deg = make_int2(0, 0);
    if (da != kInf) {
      ib = c.ib[2 * int64_t(da)];
      deg = reinterpret_cast<const int2*>(c.dslot)[da];
    }
    for (int64_t q0 = b0; q0 < b1; q0 += 32) {
      const int64_t q = q0 + lane;
      Msg m;
      m.a = ida;
      m.ta = ta;
      const int32_t pb = q < b1 ? col[q] : 0;
      const bool has = q < b1 && pb > a;
      m.tb = has ? c.first_slot[pb] : kInf;
      m.b = has ? c.order[pb] : 0;
      m.d = min(da, trade_of(m.tb));
      const bool mine = has && da != kInf && m.d == da && trade_of(m.tb) != da && da != c.hold_trade;
      const unsigned mm = __ballot_sync(kFull, mine);
      if (mm) {
        const unsigned long long one = (ta & 1) ? (1ull << 32) : 1ull;
        unsigned long long old = 0;
        if (lane == 0) old = atomicAdd(&c.fill[da], one * static_cast<unsigned>(__popc(mm)));
        old = __shfl_sync(kFull, old, 0);
        m.old = old + one * static_cast<unsigned>(__popc(mm & ((1u << lane) - 1u)));
        m.ib = ib;
        m.deg = deg;
        if (mine) deliver(c, m);
      }
      // hold_trade is a test hook: messages to that trade are dropped, so it never becomes runnable
      if (has && !mine && !(m.d == c.hold_trade)) {
        reserve(c, m);
        deliver(c, m);
      }
    }
  }
  for (int64_t k = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; k < c.L; k += int64_t(gridDim.x) * blockDim.x)
    if (c.dslot[2 * k] == 0 && c.dslot[2 * k + 1] == 0) push(c, k, 0);
}

// Bounded wait for an inbox entry still being written (the cold path).
__device__ __noinline__ bool wait_entry(const int2* p, const int32_t* err, uint64_t wait_ns, int2* out) {
  int2 m = ld_relaxed_v2(p);
  if (m.x != -1) {
    *out = m;
    return true;
  }
  const uint64_t t0 = globaltimer();
  for (;;) {
    __nanosleep(100);
    m = ld_relaxed_v2(p);
    if (m.x != -1) {
      *out = m;
      return true;
    }
    if (ld_volatile_i32(err) != 0 || globaltimer() - t0 > wait_ns) return false;
  }
}

// Per-trade work space: the gathered entries (neighbour, its next trade),
// their shuffle keys, flags and a hash of u's neighbours.
template <class HT>
struct TradeWs {
  int2* ent;
  uint64_t* key;
  HT* hash;        // entry index + 1 of u's neighbours, 0 = empty
  uint8_t* flag;   // bit 0 side (0: u's inbox, 1: v's), bit 1 common, bit 2 the edge {u, v}, bit 3 to u
};

// Big trades keep their entries in global memory but hash u's neighbours in
// the (then unused) shared memory with 16-bit slots, up to this degree of u
// at a load factor of at most 3/4.
constexpr int kHash16MaxDu = 12288;

constexpr size_t kWsBytesPerElem = sizeof(int2) + sizeof(uint64_t) + 2 * sizeof(int32_t) + 1;

__device__ __forceinline__ TradeWs<int32_t> carve_ws(char* base, int64_t cap) {
  TradeWs<int32_t> w;
  w.ent = reinterpret_cast<int2*>(base);
  w.key = reinterpret_cast<uint64_t*>(base + sizeof(int2) * cap);
  w.hash = reinterpret_cast<int32_t*>(base + (sizeof(int2) + sizeof(uint64_t)) * cap);
  w.flag = reinterpret_cast<uint8_t*>(base + (sizeof(int2) + sizeof(uint64_t) + 2 * sizeof(int32_t)) * cap);
  return w;
}

// log2 of the smallest power of two >= max(want, 2)
__device__ __forceinline__ int hash_bits(int64_t want) {
  int b = 1;
  while ((int64_t(1) << b) < want) ++b;
  return b;
}

__device__ __forceinline__ uint32_t hash_slot(int32_t x, int hbits) {
  return (static_cast<uint32_t>(x) * 0x9E3779B1u) >> (32 - hbits);
}

// Elements of D with the same full key as entry e and a smaller node id
// (ties of 64-bit keys: practically never, hence the plain loop).
__device__ __noinline__ int tied_before(const int2* ent, const uint64_t* key, const uint8_t* flag,
                                        int E, int e) {
  const int32_t id = ent[e].x;
  int before = 0;
  for (int q = 0; q < E; ++q)
    if ((flag[q] & 6) == 0 && key[q] == key[e] && ent[q].x < id) ++before;
  return before;
}

// Trade k: its nodes, their degrees, their next slots, and its inbox (u's
// entries, then v's).  Loaded together as soon as k is known.
struct Trade {
  int2 uv, deg, next;
  const int2* in;
};

__device__ __forceinline__ Trade load_trade(const UniCtx& c, int64_t k) {
  return Trade{reinterpret_cast<const int2*>(c.tp)[k], reinterpret_cast<const int2*>(c.dslot)[k],
               reinterpret_cast<const int2*>(c.nxt)[k], c.inbox + c.ib[2 * k]};
}

// One trade by a team.  Returns false when a wait gave up.
template <class Team, class HT>
__device__ bool uni_trade(Team& tm, const UniCtx& c, int64_t k, const Trade& t, const TradeWs<HT>& w, int hbits, int32_t* hist,
                          int* s_sel, int* s_abort, unsigned long long& moved, unsigned long long& possible) {
  constexpr int NT = Team::N;
  const int32_t u = t.uv.x, v = t.uv.y;
  const int du = t.deg.x, E = t.deg.x + t.deg.y;
  const int2 next = t.next;
  const int2* in = t.in;
  const int H = 1 << hbits;
  const uint64_t gi = c.first + static_cast<uint64_t>(k);
  // 1. gather both inboxes: plain L2 loads, and a bounded wait only for an
  //    entry still in flight; trade k's shuffle keys (Philox on (node id, k));
  //    clear the hash
  bool ok = true;
#pragma unroll 4
  for (int e = tm.rank; e < E; e += NT) {
    int2 m = __ldcg(in + e);
    if (m.x == -1 && !wait_entry(in + e, c.err, c.wait_ns, &m)) {
      ok = false;
      m = make_int2(0, kInf);
    }
    const Philox4 r = philox4x32_10(static_cast<uint32_t>(m.x), static_cast<uint32_t>(gi), static_cast<uint32_t>(gi >> 32), 6u, c.seed);
    w.ent[e] = m;
    w.key[e] = (static_cast<uint64_t>(r.w0) << 32) | r.w1;
    w.flag[e] = static_cast<uint8_t>(e >= du ? (m.x == u ? 5 : 1) : (m.x == v ? 4 : 0));
  }
  for (int s = tm.rank; s < H; s += NT) w.hash[s] = 0;
  if (!ok) atomicExch(s_abort, 1);
  tm.sync();
  if (*s_abort) return false;
  // 2. u's neighbours into the hash (entry index + 1)
  for (int e = tm.rank; e < du; e += NT) {
    uint32_t s = hash_slot(w.ent[e].x, hbits);
    while (atomicCAS(&w.hash[s], HT(0), static_cast<HT>(e + 1)) != HT(0)) s = (s + 1) & (H - 1);
  }
  tm.sync();
  // 3. v's neighbours look themselves up: common neighbours
  for (int e = du + tm.rank; e < E; e += NT) {
    const int32_t x = w.ent[e].x;
    uint32_t s = hash_slot(x, hbits);
    for (;;) {
      const int32_t h = static_cast<int32_t>(w.hash[s]);
      if (h == 0) break;
      if (w.ent[h - 1].x == x) {
        w.flag[e] = 3;
        w.flag[h - 1] = 2;   // side 0, common
        break;
      }
      s = (s + 1) & (H - 1);
    }
  }
  tm.sync();
  // 4. D = the rest
  int64_t cnt = 0;
  for (int e = tm.rank; e < E; e += NT) {
    const uint8_t f = w.flag[e];
    if ((f & 6) == 0) cnt += 1 + ((f & 1) ? 0 : (int64_t(1) << 32));
  }
  cnt = tm.sum(cnt);
  const int nd = static_cast<int>(cnt & 0xffffffff), na = static_cast<int>(cnt >> 32);
  // 5. sigma(D) sorts D by (key, node id); u receives the first na (Fig. 2).
  //    Radix select of the na-th smallest key, 8 bits at a time from the top.
  uint64_t prefix = 0, mask = 0;
  int r = na;
  bool tie = false;
  if (na > 0 && na < nd) {
    for (int shift = 56;; shift -= 8) {
      for (int b = tm.rank; b < 256; b += NT) hist[b] = 0;
      tm.sync();
#pragma unroll 4
      for (int e = tm.rank; e < E; e += NT)
        if ((w.flag[e] & 6) == 0 && (w.key[e] & mask) == prefix) atomicAdd(&hist[(w.key[e] >> shift) & 255], 1);
      tm.sync();
      // two bins to each of the first 128 threads
      const bool bins = tm.rank < 128;
      const int h0 = bins ? hist[2 * tm.rank] : 0, h1 = bins ? hist[2 * tm.rank + 1] : 0;
      const int below = static_cast<int>(tm.exscan32(static_cast<uint32_t>(h0 + h1)));
      if (bins && below < r && r <= below + h0 + h1) {
        const int hi = r > below + h0;
        s_sel[0] = 2 * tm.rank + hi;
        s_sel[1] = hi ? h1 : h0;
        s_sel[2] = hi ? below + h0 : below;
      }
      tm.sync();
      const int b = s_sel[0], size = s_sel[1];
      r -= s_sel[2];
      prefix |= static_cast<uint64_t>(b) << shift;
      mask |= uint64_t(255) << shift;
      if (size == 1) break;
      if (shift == 0) {
        tie = true;   // several elements share the full key: node id decides
        break;
      }
    }
  }
  // 6. every resulting edge goes on: common neighbours and the edge {u, v}
  //    stay, an element of D below the threshold's bucket goes to u, above it
  //    to v, within it by rank.  One message at a time: two to four in flight
  //    cost registers and took 8 to 22 % longer.
  for (int e = tm.rank; e < E; e += NT) {
    const uint8_t f = w.flag[e];
    const int2 en = w.ent[e];
    if ((f & 5) == 5) continue;   // the edge {u, v} goes on from u's entry
    Msg m;
    bool at_u = !(f & 1);
    if (!(f & 6)) {
      if (na == 0) at_u = false;
      else if (na == nd) at_u = true;
      else {
        const uint64_t km = w.key[e] & mask;
        if (km != prefix) at_u = km < prefix;
        else if (!tie) at_u = r >= 1;   // the single element of the last bucket is the na-th
        else at_u = tied_before(w.ent, w.key, w.flag, E, e) < r;
      }
      moved += at_u == ((f & 1) != 0);   // an edge end that changes node
    }
    m.a = at_u ? u : v;
    m.ta = at_u ? next.x : next.y;
    m.b = en.x;
    m.tb = (f & 4) ? next.y : en.y;
    reserve(c, m);
    deliver(c, m);
  }
  if (tm.rank == 0) possible += static_cast<unsigned>(E);
  tm.sync();   // the work space is reused by the next trade
  return true;
}

// messages of a small trade's lane with their atomics in flight together
constexpr int kMsgBatch = 2;
constexpr int kSmallHash = 2 * kUniSmall;   // hash slots of a small trade's work space
constexpr int32_t kMark = static_cast<int32_t>(0x80000000u);

// A small trade (E <= 32 J) by a warp: entry 32 j + lane in register j,
// u's neighbours hashed by position (-1: empty; top bit: v has it too), the
// threshold found bit by bit, about log2 |D| + 2 votes.  Its latency is what
// counts, hence a form each for J = 1, 2 and 4.
template <int J>
__device__ __noinline__ bool uni_trade_warp(const UniCtx& c, int64_t k, Trade t, int32_t* hash, unsigned long long& moved,
                               unsigned long long& possible) {
  constexpr int kBatch = J < kMsgBatch ? J : kMsgBatch;
  static_assert(J % kBatch == 0, "");
  const int lane = threadIdx.x & 31;
  const int32_t u = t.uv.x, v = t.uv.y;
  const int du = t.deg.x, E = t.deg.x + t.deg.y;
  const int2 next = t.next;
  const int2* in = t.in;
  const int hbits = hash_bits(2 * du);
  const int H = 1 << hbits;
  const uint64_t gi = c.first + static_cast<uint64_t>(k);
  int2 m[J];
  bool ok = true;
#pragma unroll
  for (int j = 0; j < J; ++j) m[j] = 32 * j + lane < E ? __ldcg(in + 32 * j + lane) : make_int2(-2, kInf);
  for (int s = lane; s < H; s += 32) hash[s] = -1;
#pragma unroll
  for (int j = 0; j < J; ++j)
    if (m[j].x == -1 && !wait_entry(in + 32 * j + lane, c.err, c.wait_ns, &m[j])) {
      ok = false;
      m[j] = make_int2(0, kInf);
    }
  if (__any_sync(kFull, !ok)) return false;
  __syncwarp();
  uint64_t key[J];
  int at[J];
#pragma unroll
  for (int j = 0; j < J; ++j) {
    const int e = 32 * j + lane;
    at[j] = 0;
    if (e < du) {
      uint32_t s = hash_slot(m[j].x, hbits);
      while (atomicCAS(&hash[s], -1, m[j].x) != -1) s = (s + 1) & (H - 1);
      at[j] = static_cast<int>(s);
    }
  }
  __syncwarp();
  // 0: in D, 1: stays (common neighbour), 2: the edge {u, v} or no entry
  uint32_t kind[J];
#pragma unroll
  for (int j = 0; j < J; ++j) {
    const int e = 32 * j + lane;
    kind[j] = e < E ? 0u : 2u;
    if (e >= du && e < E) {
      if (m[j].x == u) kind[j] = 2u;
      uint32_t s = hash_slot(m[j].x, hbits);
      for (;;) {
        const int32_t h = hash[s];
        if (h == -1) break;
        if ((h & ~kMark) == m[j].x) {
          kind[j] = 1u;
          hash[s] = h | kMark;
          break;
        }
        s = (s + 1) & (H - 1);
      }
    }
  }
  __syncwarp();
  uint32_t cnt = 0;   // |D| and, above bit 16, u's part of it
#pragma unroll
  for (int j = 0; j < J; ++j) {
    const int e = 32 * j + lane;
    if (e < du) {
      if (m[j].x == v) kind[j] = 2u;
      else if (hash[at[j]] < 0) kind[j] = 1u;
    }
    key[j] = 0;
    if (kind[j] == 0u) {
      const Philox4 r = philox4x32_10(static_cast<uint32_t>(m[j].x), static_cast<uint32_t>(gi),
                                      static_cast<uint32_t>(gi >> 32), 6u, c.seed);
      key[j] = (static_cast<uint64_t>(r.w0) << 32) | r.w1;
      cnt += e < du ? 0x10001u : 1u;
    }
  }
  cnt = __reduce_add_sync(kFull, cnt);
  int size = static_cast<int>(cnt & 0xffffu), r = static_cast<int>(cnt >> 16);
  // the na smallest keys of D to u: candidates share the threshold's prefix,
  // r of them are still to go to u
  uint32_t cand = 0, to_u = 0;   // bit j: entry j
#pragma unroll
  for (int j = 0; j < J; ++j) cand |= (kind[j] == 0u) << j;
  for (int bit = 63; r > 0 && r < size && bit >= 0; --bit) {
    uint32_t zero = 0;
#pragma unroll
    for (int j = 0; j < J; ++j) zero |= static_cast<uint32_t>(~(key[j] >> bit) & 1ull) << j;
    zero &= cand;
    const int z = static_cast<int>(__reduce_add_sync(kFull, __popc(zero)));
    if (r < z) {
      cand = zero;
      size = z;
    } else {
      to_u |= zero;
      cand &= ~zero;
      size -= z;
      r -= z;
    }
  }
  if (r > 0 && r < size) {   // equal full keys: node id decides (practically never)
    uint32_t id[J];
#pragma unroll
    for (int j = 0; j < J; ++j) id[j] = (cand >> j & 1u) ? static_cast<uint32_t>(m[j].x) : 0xffffffffu;
#pragma unroll
    for (int j = 0; j < J; ++j) {
      int before = 0;
      for (int q = 0; q < 32; ++q)
#pragma unroll
        for (int i = 0; i < J; ++i) before += __shfl_sync(kFull, id[i], q) < id[j];
      if ((cand >> j & 1u) && before < r) to_u |= 1u << j;
    }
  } else if (r > 0) {
    to_u |= cand;   // r == size
  }
  // every resulting edge goes on, kBatch messages of a lane in flight
  uint32_t has = 0;
#pragma unroll
  for (int j = 0; j < J; ++j) {
    const bool side_u = 32 * j + lane < du;
    if (kind[j] == 1u && side_u) to_u |= 1u << j;
    if (kind[j] == 0u) moved += (to_u >> j & 1u) != static_cast<uint32_t>(side_u);
    if (kind[j] == 2u && side_u) {   // the edge {u, v}: from u's entry only
      m[j].y = next.y;
      to_u |= 1u << j;
      kind[j] = 1u;
    }
    has |= (kind[j] != 2u) << j;
  }
#pragma unroll
  for (int j0 = 0; j0 < J; j0 += kBatch) {
    Msg msg[kBatch];
#pragma unroll
    for (int q = 0; q < kBatch; ++q) {
      const int j = j0 + q;
      const bool at_u = to_u >> j & 1u;
      msg[q].a = at_u ? u : v;
      msg[q].ta = at_u ? next.x : next.y;
      msg[q].b = m[j].x;
      msg[q].tb = m[j].y;
      if (has >> j & 1u) reserve(c, msg[q]);
    }
#pragma unroll
    for (int q = 0; q < kBatch; ++q)
      if (has >> (j0 + q) & 1u) deliver(c, msg[q]);
  }
  if (lane == 0) possible += static_cast<unsigned>(E);
  __syncwarp();   // the hash is reused by the next trade
  return true;
}

// The executor.  n=2^20, degrees [10,1000), n/2 trades: 28.8 ms with every
// trade on a whole 1024-thread CTA, 10.1 ms so: 152 trades ran at once, now
// up to 1368, and a trade has two dependent memory accesses fewer.
template <int NT>
__global__ void __launch_bounds__(NT, 1024 / NT) k_uni_exec(const __grid_constant__ UniCtx c) {
  constexpr int kTeam = uni_team<NT>();
  extern __shared__ __align__(16) char usm[];
  __shared__ int64_t red[SubTeam<kTeam>::kRedSlots];
  __shared__ int32_t hist[256];
  __shared__ int s_sel[3];
  __shared__ int64_t s_k;
  __shared__ int s_abort;
  __shared__ int32_t small_hash[uni_warps<NT>()][kSmallHash];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  unsigned long long moved = 0, possible = 0;   // swaps, for the handle's counters
  const RunQueues rq = queues(c);
  bool ok = true;
  int32_t* hash = warp < kTeam / 32 ? reinterpret_cast<int32_t*>(usm) + warp * kSmallHash : small_hash[warp - kTeam / 32];
  if (warp < kTeam / 32) {
    SubTeam<kTeam> tm(red, 0);
    if (tm.rank == 0) s_abort = 0;
    const TradeWs ws_smem = carve_ws(usm, uni_smem_elems<NT>());
    const TradeWs ws_glob =
        c.gslice ? carve_ws(c.gslice + static_cast<size_t>(blockIdx.x) * c.slice_elems * kWsBytesPerElem, c.slice_elems)
                 : ws_smem;
    while (ok) {
      if (tm.rank == 0) s_k = take_ticket(c, 1, rq);
      tm.sync();
      const int64_t k = s_k;
      if (k < 0) break;
      const Trade t = load_trade(c, k);
      const int64_t du = t.deg.x, E = du + t.deg.y;
      if (E > uni_smem_elems<NT>() && du <= kHash16MaxDu) {
        TradeWs<uint16_t> w16{ws_glob.ent, ws_glob.key, reinterpret_cast<uint16_t*>(usm), ws_glob.flag};
        ok = uni_trade(tm, c, k, t, w16, hash_bits((4 * du + 2) / 3), hist, s_sel, &s_abort, moved, possible);
      } else {
        ok = uni_trade(tm, c, k, t, E <= uni_smem_elems<NT>() ? ws_smem : ws_glob, hash_bits(2 * du), hist, s_sel, &s_abort,
                       moved, possible);
      }
    }
  }
  while (ok) {
    int64_t k = 0;
    if (lane == 0) k = take_ticket(c, 0, rq);
    k = __shfl_sync(kFull, k, 0);
    if (k < 0) break;
    const Trade t = load_trade(c, k);
    const int E = t.deg.x + t.deg.y;
    ok = E <= 32   ? uni_trade_warp<1>(c, k, t, hash, moved, possible)
         : E <= 64 ? uni_trade_warp<2>(c, k, t, hash, moved, possible)
                   : uni_trade_warp<kUniSmall / 32>(c, k, t, hash, moved, possible);
  }
  if (!ok && lane == 0) latch(c.err, kErrUniformWait);
  if (c.swaps) {
    const int64_t mv = WarpTeam().sum(static_cast<int64_t>(moved)), ps = WarpTeam().sum(static_cast<int64_t>(possible));
    if (lane == 0 && (mv | ps)) {
      atomicAdd(&c.swaps[0], static_cast<unsigned long long>(mv));
      atomicAdd(&c.swaps[1], static_cast<unsigned long long>(ps));
    }
  }
}

// Every output row full, and every place of both queues filled once and taken.
__global__ void k_uni_check(int64_t n, const int64_t* __restrict__ rp, const int32_t* __restrict__ ocur,
                            const unsigned long long* __restrict__ ctr, int64_t L, int32_t* err) {
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    const RunQueues rq{L, static_cast<int64_t>(ctr[kBig])};
    for (int big = 0; big < 2; ++big) {
      const int64_t len = rq.length(big);
      if (static_cast<int64_t>(ctr[kQueueCtr * big + kTail]) != len || static_cast<int64_t>(ctr[kQueueCtr * big + kHead]) < len)
        latch(err, kErrUniform);
    }
  }
  for (int64_t x = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; x < n; x += int64_t(gridDim.x) * blockDim.x)
    if (ocur[x] != rp[x + 1] - rp[x]) latch(err, kErrRowLength);
}

unsigned grid_for_work(int64_t work, int num_sms) {
  const int64_t want = (work + 255) / 256;
  return static_cast<unsigned>(std::max<int64_t>(1, std::min<int64_t>(want, int64_t(num_sms) * 16)));
}

template <class T>
cudaError_t grow(Graph* h, T** p, int64_t count, size_t* bytes) {
  if (count <= 0) count = 1;
  void* q = nullptr;
  const cudaError_t e = dev_alloc(h, &q, sizeof(T) * static_cast<size_t>(count));
  if (e == cudaSuccess) {
    *p = static_cast<T*>(q);
    *bytes += sizeof(T) * static_cast<size_t>(count);
  }
  return e;
}

int uni_buffers(Graph* h, int64_t L) {
  UniBufs* b = h->uni;
  if (b && b->cap_trades >= L && b->n == h->n) return CB_OK;
  free_uniform(h);
  b = new UniBufs;
  h->uni = b;
  const int64_t n = h->n;
  b->cap_trades = L;
  b->n = n;
  size_t* by = &b->bytes;
  if (grow(h, &b->tp, 2 * L, by) || grow(h, &b->dslot, 2 * L, by) || grow(h, &b->ib, 2 * L + 1, by) ||
      grow(h, &b->suc, 2 * L, by) || grow(h, &b->nxt, 2 * L, by) || grow(h, &b->fill, L, by) ||
      grow(h, &b->queue, L, by) || grow(h, &b->occ, n, by) || grow(h, &b->sbeg, n + 1, by) ||
      grow(h, &b->ocur, n, by) || grow(h, &b->first, n, by) || grow(h, &b->ctr, kCtrWords, by))
    return fail(h, CB_ENOMEM, "device allocation failed (uniform trades)");
  const size_t ws = std::max(scan_ws_bytes(n), scan_ws_bytes(2 * L));
  void* q = nullptr;
  if (dev_alloc(h, &q, ws)) return fail(h, CB_ENOMEM, "device allocation failed (uniform trades)");
  b->scan_ws = q;
  b->bytes += ws;
  return CB_OK;
}

}  // namespace

void free_uniform(Graph* h) {
  UniBufs* b = h->uni;
  if (!b) return;
  void* bufs[] = {b->tp, b->dslot, b->ib, b->suc, b->nxt, b->fill, b->queue, b->occ, b->sbeg, b->ocur, b->first, b->ctr,
                  b->scan_ws};
  if (h->stream) {
    for (void* p : bufs)
      if (p) cudaFreeAsync(p, h->stream);
    if (b->inbox) cudaFreeAsync(b->inbox, h->stream);
    if (b->gslice) cudaFreeAsync(b->gslice, h->stream);
  }
  h->dev_bytes -= static_cast<int64_t>(b->bytes + b->inbox_bytes + b->slice_bytes);
  delete b;
  h->uni = nullptr;
}

int uniform_trades(Graph* h, uint64_t count) {
  if (h->nseg != 1) return fail(h, CB_EINVAL, "uniform trades are for handles of one graph");
  const int64_t n = h->n;
  if (n < 2 || count == 0) {
    h->uni_next += count;
    return CB_OK;
  }
  cudaStream_t s = h->stream;
  const int64_t launches0 = h->launches;
  const int64_t chunk = std::max<int64_t>(n / 2, kUniChunkMin);
  int rc;
  if ((rc = uni_buffers(h, std::min<int64_t>(chunk, static_cast<int64_t>(std::min<uint64_t>(count, 1ull << 40))))))
    return rc;
  UniBufs* b = h->uni;
  // kernel resources: occupancy of the persistent executor, its sort space
  const int NT = h->uni_threads;
  const void* exec = NT == 1024 ? reinterpret_cast<const void*>(k_uni_exec<1024>)
                     : NT == 512 ? reinterpret_cast<const void*>(k_uni_exec<512>)
                                 : reinterpret_cast<const void*>(k_uni_exec<256>);
  const int smem_elems = NT == 1024 ? uni_smem_elems<1024>() : uni_smem_elems<256>();
  const size_t smem = kWsBytesPerElem * smem_elems;
  CB_CUDA(h, cudaFuncSetAttribute(exec, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(smem)));
  int per_sm = 0;
  CB_CUDA(h, cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, exec, NT, smem));
  const int ctas = std::max(1, per_sm) * h->num_sms;
  const int64_t big = next_pow2_host(std::max<int64_t>(2 * h->maxdeg, 1));
  if (2 * h->maxdeg > smem_elems && (!b->gslice || b->slice_elems < big || b->ctas < ctas)) {
    if (b->gslice) {
      cudaFreeAsync(b->gslice, s);
      h->dev_bytes -= static_cast<int64_t>(b->slice_bytes);
      b->gslice = nullptr;
      b->slice_bytes = 0;
    }
    const size_t bytes = static_cast<size_t>(big) * kWsBytesPerElem * ctas;
    void* q = nullptr;
    if (dev_alloc(h, &q, bytes)) return fail(h, CB_ENOMEM, "device allocation failed (uniform sort space)");
    b->gslice = static_cast<char*>(q);
    b->slice_elems = big;
    b->slice_bytes = bytes;
    b->ctas = ctas;
  }
  const unsigned g1 = grid_for_work(n, h->num_sms);
  uint64_t done = 0;
  while (done < count) {
    const int64_t L = static_cast<int64_t>(std::min<uint64_t>(count - done, static_cast<uint64_t>(b->cap_trades)));
    const uint64_t first = h->uni_next + done;
    const unsigned gL = grid_for_work(L, h->num_sms);
    // the sequence in positions, its Suc lists and every slot's next slot
    CB_CUDA(h, cudaMemsetAsync(b->occ, 0, sizeof(int32_t) * n, s));
    CB_CUDA(h, cudaMemsetAsync(b->ctr, 0, sizeof(unsigned long long) * kCtrWords, s));
    k_uni_draw<<<gL, 256, 0, s>>>(L, first, h->seed, n, h->deg_id, b->tp, b->dslot, b->occ, uni_small(L), b->ctr + kBig);
    CB_CUDA(h, cudaGetLastError());
    CB_CUDA(h, exclusive_scan_i32(b->occ, b->sbeg, n, b->scan_ws, s, &h->launches));
    CB_CUDA(h, cudaMemsetAsync(b->occ, 0, sizeof(int32_t) * n, s));
    k_uni_fill<<<grid_for_work(2 * L, h->num_sms), 256, 0, s>>>(2 * L, b->tp, b->sbeg, b->occ, b->suc);
    CB_CUDA(h, cudaGetLastError());
    k_uni_sort<<<g1, 256, 0, s>>>(n, b->sbeg, b->suc, b->nxt, h->pos[h->cur], b->first);
    CB_CUDA(h, cudaGetLastError());
    CB_CUDA(h, exclusive_scan_i32(b->dslot, b->ib, 2 * L, b->scan_ws, s, &h->launches));
    int64_t total = 0;
    CB_CUDA(h, cudaMemcpyAsync(&total, b->ib + 2 * L, sizeof(int64_t), cudaMemcpyDeviceToHost, s));
    CB_CUDA(h, cudaStreamSynchronize(s));
    if (total > b->inbox_cap) {
      if (b->inbox) {
        cudaFreeAsync(b->inbox, s);
        h->dev_bytes -= static_cast<int64_t>(b->inbox_bytes);
        b->inbox = nullptr;
        b->inbox_cap = 0;
        b->inbox_bytes = 0;
      }
      const int64_t cap = total + total / 8 + 1024;
      void* q = nullptr;
      if (dev_alloc(h, &q, sizeof(int2) * static_cast<size_t>(cap)))
        return fail(h, CB_ENOMEM, "device allocation failed (uniform inboxes)");
      b->inbox = static_cast<int2*>(q);
      b->inbox_cap = cap;
      b->inbox_bytes = sizeof(int2) * static_cast<size_t>(cap);
    }
    // empty inboxes (every byte 0xff: node -1), counts, queue, output cursors
    if (total) CB_CUDA(h, cudaMemsetAsync(b->inbox, 0xff, sizeof(int2) * static_cast<size_t>(total), s));
    CB_CUDA(h, cudaMemsetAsync(b->fill, 0, sizeof(unsigned long long) * L, s));
    CB_CUDA(h, cudaMemsetAsync(b->queue, 0xff, sizeof(int32_t) * L, s));
    CB_CUDA(h, cudaMemsetAsync(b->ocur, 0, sizeof(int32_t) * n, s));
    const int spare = 1 - h->cur;
    UniCtx c;
    c.L = L;
    c.first = first;
    c.seed = h->seed;
    c.rp = h->rp[h->cur];
    c.order = h->order[h->cur];
    c.tp = b->tp;
    c.nxt = b->nxt;
    c.ib = b->ib;
    c.dslot = b->dslot;
    c.pos = h->pos[h->cur];
    c.first_slot = b->first;
    c.inbox = b->inbox;
    c.fill = b->fill;
    c.queue = b->queue;
    c.ctr = b->ctr;
    c.ocur = b->ocur;
    c.col_out = h->col[spare];
    c.wait_ns = h->uni_wait_ns;
    c.small = uni_small(L);
    c.hold_trade = h->hold_trade;
    c.err = h->err;
    c.gslice = b->gslice;
    c.slice_elems = b->slice_elems;
    c.swaps = h->swap_stats ? reinterpret_cast<unsigned long long*>(h->swaps) : nullptr;
    k_uni_route<<<grid_for_work(n * 32, h->num_sms), 256, 0, s>>>(c, n, h->col[h->cur]);
    CB_CUDA(h, cudaGetLastError());
    if (NT == 1024) k_uni_exec<1024><<<ctas, 1024, smem, s>>>(c);
    else if (NT == 512) k_uni_exec<512><<<ctas, 512, smem, s>>>(c);
    else k_uni_exec<256><<<ctas, 256, smem, s>>>(c);
    CB_CUDA(h, cudaGetLastError());
    k_uni_check<<<g1, 256, 0, s>>>(n, c.rp, b->ocur, b->ctr, L, h->err);
    CB_CUDA(h, cudaGetLastError());
    h->launches += 6;
    if ((rc = check_device_error(h))) return rc;
    std::swap(h->col[h->cur], h->col[spare]);
    done += static_cast<uint64_t>(L);
  }
  h->uni_next += count;
  h->stats[5] = h->launches - launches0;
  // the recorded super steps name the old adjacency buffers; exports are stale
  drop_step_graphs(h);
  h->pairs_step = ~0ull;
  return CB_OK;
}

}  // namespace cb

extern "C" int cb_uniform_trades(cb_handle h, uint64_t count) {
  using namespace cb;
  if (!h) return fail(nullptr, CB_EINVAL, "NULL handle");
  if (h->latched) return fail(h, h->latched, "handle has a latched error: " + h->last_error);
  return uniform_trades(h, count);
}

extern "C" int cb_uniform_next(cb_handle h, uint64_t* next) {
  using namespace cb;
  if (!h || !next) return fail(h, CB_EINVAL, "bad argument");
  *next = h->uni_next;
  return CB_OK;
}

extern "C" int cb_uniform_pairs(uint64_t seed, int64_t n, uint64_t first, int64_t count, int32_t* pairs,
                                void* cuda_stream) {
  using namespace cb;
  if (n < 2 || n > 0x7fffffffLL || count < 0 || (count > 0 && !pairs))
    return fail(nullptr, CB_EINVAL, "cb_uniform_pairs: needs 2 <= n < 2^31, count >= 0 and a buffer");
  if (count == 0) return CB_OK;
  int dev = 0, num_sms = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&num_sms, cudaDevAttrMultiProcessorCount, dev);
  if (e != cudaSuccess) return cuda_fail(nullptr, e, "device query");
  cudaStream_t s = static_cast<cudaStream_t>(cuda_stream);
  k_uni_draw<<<grid_for_work(count, num_sms), 256, 0, s>>>(count, first, seed, n, nullptr, pairs, nullptr, nullptr, 0, nullptr);
  if ((e = cudaGetLastError()) != cudaSuccess) return cuda_fail(nullptr, e, "k_uni_draw");
  return CB_OK;
}

extern "C" int cb_successors(int64_t n, const int32_t* pairs, int64_t count, int64_t* suc_begin, int32_t* suc,
                             void* cuda_stream) {
  using namespace cb;
  if (n < 0 || n > 0x7fffffffLL || count < 0 || count > 0x3fffffffLL || !suc_begin || (count > 0 && (!pairs || !suc)))
    return fail(nullptr, CB_EINVAL, "cb_successors: bad n, count or buffer");
  int dev = 0, num_sms = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&num_sms, cudaDevAttrMultiProcessorCount, dev);
  if (e != cudaSuccess) return cuda_fail(nullptr, e, "device query");
  cudaStream_t s = static_cast<cudaStream_t>(cuda_stream);
  // scratch: occurrence counts / cursors, slot lists, an error word, scan space
  const size_t ws = scan_ws_bytes(n);
  const size_t bytes = sizeof(int32_t) * (static_cast<size_t>(n) + 2 * static_cast<size_t>(count) + 1) + ws + 16;
  char* scratch = nullptr;
  if ((e = cudaMallocAsync(reinterpret_cast<void**>(&scratch), bytes, s)) != cudaSuccess)
    return cuda_fail(nullptr, e, "cudaMallocAsync");
  int32_t* occ = reinterpret_cast<int32_t*>(scratch);
  int32_t* slots = occ + n;
  int32_t* err = slots + 2 * count;
  void* scan = scratch + ((sizeof(int32_t) * (n + 2 * count + 1) + 15) & ~size_t(15));
  int rc = CB_OK;
  int32_t herr = 0;
  const unsigned g = grid_for_work(std::max<int64_t>(n, 2 * count), num_sms);
  if ((e = cudaMemsetAsync(occ, 0, sizeof(int32_t) * (n + 2 * count + 1), s)) != cudaSuccess) goto cuda_error;
  if (count) {
    k_uni_count<<<g, 256, 0, s>>>(count, n, pairs, occ, err);
    if ((e = cudaGetLastError()) != cudaSuccess) goto cuda_error;
  }
  if ((e = cudaMemcpyAsync(&herr, err, sizeof(int32_t), cudaMemcpyDeviceToHost, s)) != cudaSuccess) goto cuda_error;
  if ((e = cudaStreamSynchronize(s)) != cudaSuccess) goto cuda_error;
  if (herr) {
    rc = fail(nullptr, CB_EINVAL, "cb_successors: a node outside [0, n) or a pair of equal nodes");
    goto done;
  }
  if ((e = exclusive_scan_i32(occ, suc_begin, n, scan, s)) != cudaSuccess) goto cuda_error;
  if (count) {
    if ((e = cudaMemsetAsync(occ, 0, sizeof(int32_t) * n, s)) != cudaSuccess) goto cuda_error;
    k_uni_fill<<<g, 256, 0, s>>>(2 * count, pairs, suc_begin, occ, slots);
    if ((e = cudaGetLastError()) != cudaSuccess) goto cuda_error;
    k_uni_sort<<<g, 256, 0, s>>>(n, suc_begin, slots, nullptr, nullptr, nullptr);
    if ((e = cudaGetLastError()) != cudaSuccess) goto cuda_error;
    k_uni_trade_index<<<g, 256, 0, s>>>(2 * count, slots, suc);
    if ((e = cudaGetLastError()) != cudaSuccess) goto cuda_error;
  }
  if ((e = cudaStreamSynchronize(s)) != cudaSuccess) goto cuda_error;
  goto done;
cuda_error:
  rc = cuda_fail(nullptr, e, "cb_successors");
done:
  cudaFreeAsync(scratch, s);
  return rc;
}

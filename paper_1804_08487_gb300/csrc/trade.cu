// One global trade (Def. "Undirected Global Trade", Section 3.3) on the GPU.
//
// Layout: during super step g the graph is stored in position space -- row p
// holds the node at position p of the step's permutation and every entry is
// the neighbour's position (rows are sets; their order is not significant).
// Trade t owns rows 2t (u_t) and 2t+1 (v_t); the neighbour at position y
// belongs to trade y>>1.
//
// Edges joining trades s and t form a "block" of at most four edges.  A later
// trade t depends on an earlier trade s only when the block has at least two
// edges and one of t's nodes is adjacent to exactly one of s's nodes: only then
// can s's choice turn a disjoint neighbour of t into a common one or back.
// Everything else is independent, because each shuffle key belongs to an edge
// (its endpoints' positions at the start of the step), not to a node.  So a
// super step runs in two phases:
//
//  A. Threshold and placement.  Every trade finds
//     D = (A_u u A_v) \ (A_u n A_v) \ {u, v} (Def. "Simple Undirected Trade"),
//     keys its elements and publishes the threshold (key, lo, hi) of its
//     |A_{u-v}|-th smallest element: u keeps exactly the elements at or below
//     it (Fig. 2: u receives the first |A_{u-v}| elements of sigma(D)).  In
//     the same pass it places every entry in the row of its node after the
//     trade (step g+1 layout): the far end's step-g position as a placeholder,
//     and a 16-bit side word (bit 0 the own trade's flip, bits 1..11 the top
//     11 bits of the far trade's key for the edge, bit 12 set when the far
//     trade decides the edge).  The first pass runs every trade by size
//     class; a trade whose dependency has not published is deferred, retry
//     passes (large handles) run lists of them, and one in-order pass
//     completes what is left, waiting (bounded) for its dependencies.
//  B. Rebuild (fix-up).  Every placeholder becomes the step-(g+1) position
//     of the far end: per far trade one packed record (the new positions of
//     its two nodes, the top 8 bits of its threshold), read in slices small
//     enough to stay in L2; the 8-bit prefix decides, then the 11-bit one,
//     and only on a tie there the full key.
//
// Phase A by trade size L = deg u + deg v (nine classes): lane teams of 8 or
// 16 threads (several trades per warp) and whole warps up to `tile_max`
// entries, teams of 64 to 1024 threads with the entries in registers up to
// min(8192, `smem_max`), and a 1024-thread CTA with the hash in shared memory
// and the rest in a global-memory slice for the largest.  The team
// and shared-memory kernels come in a version for handles of one graph,
// whose seed's Philox round keys are kernel parameters, and a general one.
#include <algorithm>
#include <type_traits>

#include "cb_internal.cuh"
#include "classes.cuh"
#include "philox.cuh"
#include "team.cuh"

namespace cb {
namespace {

// meta bits per entry (phase A)
constexpr uint8_t kR = 1;       // entry sits in v's row
constexpr uint8_t kInD = 2;     // element of D_t
constexpr uint8_t kFlip = 4;    // trade t moves the edge to its other node
constexpr uint8_t kUV = 8;      // the edge {u_t, v_t}
// (kCol and kPend below: the neighbour's column, not hashed yet)

constexpr int kMedThreads = 256;
constexpr int kBigThreads = 1024;

struct StepCtx {
  int64_t n, T, ntasks;
  const Seg* segs;          // per graph: seed, step, first position
  const int32_t* seg_of;    // graph of each position (null: one graph)
  const int64_t* rp;
  const int32_t* col;
  uint16_t* fb;             // side word of every placed entry (step g+1 layout)
  int32_t* ph;              // placeholders of every entry in its new row (step g+1 layout)
  const int32_t* order;     // node at each position of step g
  const int32_t* pos;       // position of each node in step g
  const int32_t* order_next;   // and in step g+1
  const int32_t* pos_next;
  const int64_t* rp_next;
  const int32_t* chunk_row;    // of rp_next
  uint64_t* thr_key;
  uint64_t* thr_tb;
  void* far_pack;           // per trade: new positions of its nodes, threshold prefix (FarTrade)
  uint32_t* done;           // per trade: g + 1 once its threshold is published (only if a later trade may wait)
  int32_t* err;
  uint32_t* def_bits;              // bit t: trade t is deferred
  unsigned long long* def_n;       // trades this pass deferred, by kind
  int32_t* def_list;               // their lists by kind (pair_lists.cuh), or null: in def_bits and def_seg
  int32_t* def_seg;                // and per segment of the trades (kDefKinds x kDefSegs)
  int64_t def_seg_trades;          // trades of a segment
  int narrow;                      // 8-byte far-trade records
  unsigned long long* gws_count;
  int cand_max;                    // register paths: most candidates ranked directly (else more radix digits)
  uint64_t wait_ns;                // longest single wait on dependencies or a bulk copy
  int hold_publish;                // test hook: no trade publishes its done flag (waits run out)
  unsigned inorder_ctas;           // CTAs of the in-order pass that take part (a test hook; default: all)
  uint64_t seed;                   // one graph (seg_of null): its seed
  uint32_t ks[20];                 // and the seed's Philox round keys
};

struct SelOut {
  uint64_t key, tb;
  int32_t bin, below, cnt, pad;
};

// The trades of class k.
struct ClassList {
  const int32_t* first;
  int64_t len;
  int step;   // lists of odd classes run backwards (pair_lists.cuh)
  __device__ __forceinline__ int32_t operator[](int64_t q) const { return first[step * q]; }
};
__device__ __forceinline__ ClassList class_list(const StepCtx& c, const int32_t* lists, const int64_t* ctr, int k) {
  return {lists + pair_place(k, 0, c.ntasks), ctr[kCtrClsLen + k], (k & 1) ? -1 : 1};
}

struct TradeRows {
  int64_t b0;
  int du, dv;
  bool single;   // odd n: the untraded node at the last position
};

__device__ __forceinline__ TradeRows trade_rows(const StepCtx& c, int64_t t) {
  TradeRows r;
  r.b0 = c.rp[2 * t];
  const int64_t b1 = c.rp[2 * t + 1];
  r.single = (2 * t + 1 >= c.n);
  const int64_t b2 = r.single ? b1 : c.rp[2 * t + 2];
  r.du = static_cast<int>(b1 - r.b0);
  r.dv = static_cast<int>(b2 - b1);
  return r;
}

__device__ __forceinline__ uint32_t ld_acquire(const uint32_t* p) {
  uint32_t v;
  asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ void st_release(uint32_t* p, uint32_t v) {
  asm volatile("st.release.gpu.global.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}
__device__ __forceinline__ void latch(int32_t* err, int32_t code) { atomicCAS(err, 0, code); }
__device__ __forceinline__ uint64_t globaltimer() {
  uint64_t v;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(v));
  return v;
}
__device__ __forceinline__ int32_t ld_volatile_i32(const int32_t* p) {
  return *reinterpret_cast<const volatile int32_t*>(p);
}

// A trade whose dependency has not published, by the team that will run it
// next: listed for a retry pass, or its bit set and counted per segment for
// the in-order pass.
constexpr int kDefKinds = 3;
constexpr int kDefSmall = 128, kDefMedium = 1024;   // largest L of a warp, of 256 threads; larger: a CTA
__device__ __forceinline__ int def_kind(int L) { return L <= kDefSmall ? 0 : L <= kDefMedium ? 1 : 2; }
__device__ __forceinline__ void defer_trade(const StepCtx& c, int64_t t) {
  const TradeRows tr = trade_rows(c, t);
  const int k = def_kind(tr.du + tr.dv);
  const int64_t at = static_cast<int64_t>(atomicAdd(c.def_n + k, 1ull));
  if (c.def_list) {
    c.def_list[pair_place(k, at, c.ntasks)] = static_cast<int32_t>(t);
  } else {
    atomicOr(c.def_bits + (t >> 5), 1u << (t & 31));
    atomicAdd(c.def_seg + k * kDefSegs + t / c.def_seg_trades, 1);
  }
}

// Wait until trade s has published (true), at most wait_ns; a wait that runs
// out latches kErrResolve, and after any error every wait gives up at once.
__device__ __noinline__ bool wait_published(const uint32_t* done_s, int32_t* err, uint32_t stamp, uint64_t wait_ns) {
  const uint64_t t0 = globaltimer();
  while (ld_acquire(done_s) != stamp) {
    if (ld_volatile_i32(err) != 0) return false;
    if (globaltimer() - t0 > wait_ns) {
      latch(err, kErrResolve);
      return false;
    }
    __nanosleep(64);
  }
  return true;
}

// ------------------------------------------------- bulk copies (TMA engine)
//
// A trade's entries are staged into shared memory by one cp.async.bulk copy
// that completes on an mbarrier.  The copy moves whole 16-byte units, so it
// starts at the entry rounded down to a multiple of 4 and covers a multiple
// of 4 entries; the adjacency buffers carry 16 spare entries at their end, so
// the copy never leaves its allocation.


__device__ __forceinline__ uint32_t smem_u32(const void* p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}
__device__ __forceinline__ void mbar_init(uint64_t* m, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(m)), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_fence_init() { asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory"); }
__device__ __forceinline__ void fence_proxy_async() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }
__device__ __forceinline__ void mbar_expect_tx(uint64_t* m, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(m)), "r"(bytes) : "memory");
}
__device__ __forceinline__ void bulk_g2s(void* dst, const void* src, uint32_t bytes, uint64_t* m) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                   smem_u32(dst)),
               "l"(src), "r"(bytes), "r"(smem_u32(m))
               : "memory");
}
__device__ __forceinline__ bool mbar_test_wait(uint64_t* m, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n .reg .pred p;\n mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}"
      : "=r"(ok)
      : "r"(smem_u32(m)), "r"(parity)
      : "memory");
  return ok != 0;
}
// Bounded wait for phase `parity` of m (non-blocking polls with a short
// sleep, at most wait_ns); false if it did not complete.
__device__ __forceinline__ bool mbar_wait(uint64_t* m, uint32_t parity, uint64_t wait_ns) {
  if (mbar_test_wait(m, parity)) return true;
  const uint64_t t0 = globaltimer();
  for (;;) {
    __nanosleep(64);
    if (mbar_test_wait(m, parity)) return true;
    if (globaltimer() - t0 > wait_ns) return false;
  }
}

// Entries [b0, b0 + L) of col staged at buf + stage_off(b0).
__device__ __forceinline__ int stage_off(int64_t b0) { return static_cast<int>(b0 & 3); }
__device__ __forceinline__ void stage_issue(const int32_t* col, int64_t b0, int L, int32_t* buf, uint64_t* m) {
  const int64_t a0 = b0 & ~int64_t(3);
  const uint32_t bytes = static_cast<uint32_t>(((b0 + L - a0) + 3) & ~int64_t(3)) * 4u;
  fence_proxy_async();   // earlier generic reads of buf come before the copy's writes
  mbar_expect_tx(m, bytes);
  bulk_g2s(buf, col + a0, bytes, m);
}

__device__ __forceinline__ uint64_t tie_break(uint32_t lo, uint32_t hi) {
  return (static_cast<uint64_t>(lo) << 32) | hi;
}
// (key, tb) <= (tk, tt), lexicographic
__device__ __forceinline__ bool at_or_below(uint64_t key, uint64_t tb, uint64_t tk, uint64_t tt) {
  return key < tk || (key == tk && tb <= tt);
}

// Key parameters of a trade's graph: its seed, its step and its first
// position (keys count positions from the start of the graph).  Both ends of
// an edge are in the same graph.  kOneSeed (a handle of one graph, which starts
// at position 0): only the step is loaded, and two subtractions per edge fall
// away.  (Plain loads stay in the loop over the trades, see after_previous():
// with all three loaded per trade the in-order pass took 65.6 us at n=2^17 and
// 80 at n=2^20, n=4096 stepped ten times 597; so, 58.7, 72 and 581.)
struct KeyCtx {
  uint64_t seed;
  uint32_t g, off;
};
template <bool kOneSeed>
__device__ __forceinline__ KeyCtx key_ctx(const StepCtx& c, int64_t t) {
  if constexpr (kOneSeed) return {c.seed, c.segs->g, 0u};
  const Seg* S = c.segs + (c.seg_of ? c.seg_of[2 * t] : 0);
  return {S->seed, S->g, static_cast<uint32_t>(S->off)};
}

// Both trades' keys of the edge whose step-start positions are lo < hi.
// kOneSeed: a handle of one graph, whose seed's round keys are c.ks.
struct EdgeKeys {
  uint64_t lo_side, hi_side;
};
template <bool kOneSeed>
__device__ __forceinline__ EdgeKeys edge_keys(const StepCtx& c, const KeyCtx& kc, uint32_t lo, uint32_t hi) {
  Philox4 r;
  if constexpr (kOneSeed) {
    r = philox4x32_10_rk(lo - kc.off, hi - kc.off, kc.g, 1u, c.ks);
  } else {
    r = philox4x32_10(lo - kc.off, hi - kc.off, kc.g, 1u, kc.seed);
  }
  return {(static_cast<uint64_t>(r.w0) << 32) | r.w1, (static_cast<uint64_t>(r.w2) << 32) | r.w3};
}
__device__ __forceinline__ uint64_t side_key(const KeyCtx& kc, uint32_t lo, uint32_t hi, bool lo_side) {
  return edge_key(kc.seed, lo - kc.off, hi - kc.off, kc.g, lo_side);
}

// Does trade s send the edge (lo, hi) to its node at position 2s?  Full test.
__device__ __forceinline__ bool far_keeps_low(const StepCtx& c, const KeyCtx& kc, int64_t s, uint32_t lo,
                                              uint32_t hi) {
  const uint64_t k = side_key(kc, lo, hi, (lo >> 1) == static_cast<uint32_t>(s));
  return at_or_below(k, tie_break(lo, hi), __ldcg(c.thr_key + s), __ldcg(c.thr_tb + s));
}

// What the rebuild needs of a far trade s: the new positions of its two nodes
// and the top 8 bits of its threshold key.  Up to 2^28 positions
// (kNarrowPackMax) it fits 8 bytes (28 + 28 + 8 bits), else 16.

// Trade t's threshold, its record, and (when a later trade may wait for it)
// its done flag: by one member, as soon as the threshold is known, so that
// dependent trades wait for the threshold search and not for the placement.
// pu, pv: the positions of its nodes in step g+1.
__device__ __forceinline__ void publish(const StepCtx& c, const KeyCtx& kc, int64_t t, uint32_t pu, uint32_t pv,
                                        uint64_t tk, uint64_t tt, bool dependents) {
  c.thr_key[t] = tk;
  c.thr_tb[t] = tt;
  const uint32_t top = static_cast<uint32_t>(tk >> 56);
  if (c.narrow) {
    static_cast<uint64_t*>(c.far_pack)[t] = uint64_t(pu) | (uint64_t(pv) << 28) | (uint64_t(top) << 56);
  } else {
    static_cast<int4*>(c.far_pack)[t] =
        make_int4(static_cast<int32_t>(pu), static_cast<int32_t>(pv), static_cast<int32_t>(top), 0);
  }
  if (dependents && !c.hold_publish) {
    __threadfence();
    st_release(c.done + t, kc.g + 1u);
  }
}

// ------------------------------------------------------------ hash table
//
// One slot per far trade s of the current trade: key s + 1 (0 = empty) and a
// flag byte: bit (2 rho + gamma) = the trade's node at row rho (0: u, 1: v) is
// adjacent to s's node at position 2s + gamma (the 2x2 block matrix), bit
// (4 + 2 rho + gamma) = that entry is moved by the trade (its flip).

__device__ __forceinline__ uint32_t hslot(uint32_t s, int lgH) { return (s * 0x9E3779B1u) >> (32 - lgH); }

__device__ __forceinline__ void flag_or(uint8_t* fl, int p, uint32_t bits) {
  atomicOr(reinterpret_cast<unsigned int*>(fl + (p & ~3)), bits << (8 * (p & 3)));
}

// Slot of key (far trade + 1) starting the probe at p: the key's slot if an
// entry of the same far trade placed it, else the first empty slot, claimed
// with a compare-and-swap.  Used only for the few entries that lost the
// plain-store round of an insert.
__device__ __forceinline__ uint32_t h_claim(uint32_t* hk, uint32_t mask, uint32_t key, uint32_t p) {
  for (;;) {
    uint32_t cur = hk[p];
    if (cur == 0u) {
      cur = atomicCAS(&hk[p], 0u, key);
      if (cur == 0u) return p;
    }
    if (cur == key) return p;
    p = (p + 1u) & mask;
  }
}

// ---------------------------------------------------------- workspace

constexpr int kSelBits = 10;              // first radix digit: top 10 bits of the key
constexpr int kSelBins = 1 << kSelBits;

// meta bits per entry (team paths add the neighbour's column bit)
constexpr uint8_t kCol = 16;    // neighbour sits at the odd position 2s+1
constexpr uint8_t kPend = 32;   // not placed in the hash yet
// Bits of the far trade's key an entry's side word keeps (the rebuild decides
// with them unless they equal the far threshold's, 1 in 2^kFarBits).
constexpr int kFarBits = 11;
// Placeholder and side-word bits (see the rebuild's fix-up).
constexpr uint32_t kPhDone = 0x80000000u;   // placeholder resolved by an earlier pass (new position in bits 0..30)
constexpr uint32_t kFbInFar = 1u << 12;     // side word: the far trade decides the edge

constexpr int kCand = 32;       // candidates sharing the threshold's bin, ranked by full key

struct WsA {
  uint64_t* ck;               // kCand candidate keys
  uint64_t* ctb;              // their tie-breaks
  int32_t* cidx;              // their entry indices
  int32_t* ncand;
  int32_t* slot;              // hash slot of the entry's far trade (-1: the edge {u,v})
  uint16_t* top;              // top 16 bits of the own key
  uint8_t* meta;
  uint16_t* far;              // top kFarBits bits of the far trade's key
  uint32_t* hkey;             // 2^lgH slot keys
  uint8_t* hflag;             // 2^lgH slot flag bytes
  uint32_t* hist;             // kSelBins bins
  int lgH;
};

// table of at least twice the entries: probing always ends at an empty slot
__host__ __device__ inline int hash_lg(int L) {
  int lg = 1;
  while ((1 << lg) < 2 * L) ++lg;
  return lg;
}
__host__ __device__ inline size_t ws_a_bytes(int L) {
  const size_t L16 = (static_cast<size_t>(L) + 15) & ~size_t(15);
  const size_t H = size_t(1) << hash_lg(L);
  return H * 4 + ((H + 15) & ~size_t(15)) + kSelBins * 4 + kCand * 20 + 16 + L16 * 4 + L16 * 2 + L16 + L16 * 2 + 64;
}
// Dynamic shared memory of k_phase_a_block: workspace for `cap` entries, then
// the staging buffer of a trade's entries.
inline size_t block_smem_bytes(int cap) {
  return ((ws_a_bytes(cap) + 127) & ~size_t(127)) + (static_cast<size_t>(cap) + 8) * 4;
}

// Trades above the shared-memory cap: the hash, which every member reaches
// into, stays in shared memory while it has at most 2^kSplitLg slots (at least
// 1.25 per entry: 26214 entries), with the entries' key prefixes and flags
// while they fit; slots and far keys, which only their own member reads, go to
// the CTA's global slice.  One 1024-thread CTA per SM has the room; below, all
// of it is in the slice.  n=300007 with hubs of 15000 neighbours, everything
// above 8192 entries in the slice: first pass of the largest class 395 to 428
// us, in-order pass 1300 to 1730; so, and with the threshold published before
// the decisions: 240 to 290, and 530 to 720.
constexpr int kSplitLg = 15;
constexpr size_t kSplitSmem = size_t(224) * 1024;
__device__ inline WsA carve_split(char* smem, size_t room, char* slice, int L) {
  const size_t L16 = (static_cast<size_t>(L) + 15) & ~size_t(15);
  WsA w;
  w.lgH = hash_lg(L);
  if (w.lgH > kSplitLg && 5 * static_cast<int64_t>(L) <= (int64_t(4) << kSplitLg)) w.lgH = kSplitLg;
  const size_t H = size_t(1) << w.lgH;
  const size_t hash = H * 4 + ((H + 15) & ~size_t(15)) + kSelBins * 4 + kCand * 20 + 16;
  char* p = hash <= room ? smem : slice;
  w.hkey = reinterpret_cast<uint32_t*>(p); p += H * 4;
  w.hflag = reinterpret_cast<uint8_t*>(p); p += (H + 15) & ~size_t(15);
  w.hist = reinterpret_cast<uint32_t*>(p); p += kSelBins * 4;
  w.ck = reinterpret_cast<uint64_t*>(p); p += kCand * 8;
  w.ctb = reinterpret_cast<uint64_t*>(p); p += kCand * 8;
  w.cidx = reinterpret_cast<int32_t*>(p); p += kCand * 4;
  w.ncand = reinterpret_cast<int32_t*>(p); p += 16;
  if (hash <= room && hash + 3 * L16 > room) p = slice;
  w.top = reinterpret_cast<uint16_t*>(p); p += L16 * 2;
  w.meta = reinterpret_cast<uint8_t*>(p); p += L16;
  if (hash + 3 * L16 <= room) p = slice;
  w.slot = reinterpret_cast<int32_t*>(p); p += L16 * 4;
  w.far = reinterpret_cast<uint16_t*>(p);
  return w;
}

__device__ inline WsA carve_a(void* base, int L) {
  const size_t L16 = (static_cast<size_t>(L) + 15) & ~size_t(15);
  char* p = static_cast<char*>(base);
  WsA w;
  w.lgH = hash_lg(L);
  const size_t H = size_t(1) << w.lgH;
  w.hkey = reinterpret_cast<uint32_t*>(p); p += H * 4;
  w.hflag = reinterpret_cast<uint8_t*>(p); p += (H + 15) & ~size_t(15);
  w.hist = reinterpret_cast<uint32_t*>(p); p += kSelBins * 4;
  w.ck = reinterpret_cast<uint64_t*>(p); p += kCand * 8;
  w.ctb = reinterpret_cast<uint64_t*>(p); p += kCand * 8;
  w.cidx = reinterpret_cast<int32_t*>(p); p += kCand * 4;
  w.ncand = reinterpret_cast<int32_t*>(p); p += 16;
  w.slot = reinterpret_cast<int32_t*>(p); p += L16 * 4;
  w.top = reinterpret_cast<uint16_t*>(p); p += L16 * 2;
  w.meta = reinterpret_cast<uint8_t*>(p); p += L16;
  w.far = reinterpret_cast<uint16_t*>(p);
  return w;
}

__device__ __forceinline__ uint32_t lo_of(int64_t t2, uint8_t m, int32_t y) {
  return min(static_cast<uint32_t>(t2 + (m & kR)), static_cast<uint32_t>(y));
}
__device__ __forceinline__ uint32_t hi_of(int64_t t2, uint8_t m, int32_t y) {
  return max(static_cast<uint32_t>(t2 + (m & kR)), static_cast<uint32_t>(y));
}
__device__ __forceinline__ uint64_t own_key(const KeyCtx& kc, int64_t t, uint32_t lo, uint32_t hi) {
  return side_key(kc, lo, hi, (lo >> 1) == static_cast<uint32_t>(t));
}
// The neighbour position of a team-path entry (its far trade from the hash).
__device__ __forceinline__ int32_t entry_y(const WsA& w, int64_t t2, int i) {
  const uint8_t m = w.meta[i];
  if (m & kUV) return static_cast<int32_t>(t2 + 1 - (m & kR));
  const uint32_t s = w.hkey[w.slot[i]] - 1u;
  return static_cast<int32_t>(2 * s + ((m & kCol) ? 1 : 0));
}

// One radix digit of the 16-bit key prefixes: histogram of bits
// [shift, shift + bits) over the elements of D whose bits above equal `pre`
// (all of D when shift + bits == 16), then the bin holding the kk-th element.
template <class Team>
__device__ void radix_digit(Team& tm, const WsA& w, int L, int shift, int bits, uint32_t pre, int kk, SelOut* out) {
  const int nb = 1 << bits;
  const int bpm = (nb + Team::N - 1) / Team::N;
  for (int b = tm.rank; b < nb; b += Team::N) w.hist[b] = 0;
  tm.sync();
  for (int i = tm.rank; i < L; i += Team::N) {
    if (!(w.meta[i] & kInD)) continue;
    const uint32_t tp = w.top[i];
    if (shift + bits == 16 || (tp >> (shift + bits)) == pre) atomicAdd(&w.hist[(tp >> shift) & (nb - 1)], 1u);
  }
  tm.sync();
  const int b0 = tm.rank * bpm;
  int local = 0;
  for (int j = 0; j < bpm; ++j)
    if (b0 + j < nb) local += static_cast<int>(w.hist[b0 + j]);
  int below = static_cast<int>(tm.exscan(local));
  for (int j = 0; j < bpm; ++j) {
    const int b = b0 + j;
    if (b < nb) {
      const int hc = static_cast<int>(w.hist[b]);
      if (below < kk && kk <= below + hc) {
        out->bin = b;
        out->below = below;
        out->cnt = hc;
      }
      below += hc;
    }
  }
  tm.sync();
}

// k-th smallest (1-based) (key, lo, hi) over D, the general procedure (used
// when more than kCand elements share the threshold's bin): one 10-bit radix digit on the
// stored 16-bit key prefixes (keys are uniform, so the chosen bin holds about
// |D|/1024 elements), a 6-bit digit only if that bin is crowded, then the
// full keys of the few remaining candidates.
template <class Team>
__device__ void select_kth(Team& tm, const KeyCtx& kc, const WsA& w, int L, int64_t t, int k, SelOut* out) {
  const int64_t t2 = 2 * t;
  radix_digit(tm, w, L, 16 - kSelBits, kSelBits, 0, k, out);
  uint32_t prefix = static_cast<uint32_t>(out->bin);   // of the top `plen` bits
  int plen = kSelBits;
  int kk = k - out->below;
  int cnt = out->cnt;
  tm.sync();
  if (cnt > kCand) {
    radix_digit(tm, w, L, 0, 16 - kSelBits, prefix, kk, out);
    prefix = (prefix << (16 - kSelBits)) | static_cast<uint32_t>(out->bin);
    plen = 16;
    kk -= out->below;
    cnt = out->cnt;
    tm.sync();
  }
  uint64_t* ck = reinterpret_cast<uint64_t*>(w.hist);
  uint64_t* ctb = ck + kCand;
  int* ncand = reinterpret_cast<int*>(ctb + kCand);
  if (cnt > 1 && cnt <= kCand) {
    if (tm.rank == 0) *ncand = 0;
    tm.sync();
  }
  for (int i = tm.rank; i < L; i += Team::N) {
    const uint8_t m = w.meta[i];
    if (!(m & kInD)) continue;
    if ((static_cast<uint32_t>(w.top[i]) >> (16 - plen)) != prefix) continue;
    const int32_t y = entry_y(w, t2, i);
    const uint32_t lo = lo_of(t2, m, y), hi = hi_of(t2, m, y);
    const uint64_t ki = own_key(kc, t, lo, hi), tbi = tie_break(lo, hi);
    if (cnt == 1) {            // the only element with this prefix
      out->key = ki;
      out->tb = tbi;
    } else if (cnt <= kCand) {
      const int q = atomicAdd(ncand, 1);
      ck[q] = ki;
      ctb[q] = tbi;
    } else {                   // many equal 16-bit prefixes: rank against every other candidate
      int r = 0;
      for (int j = 0; j < L; ++j) {
        const uint8_t mj = w.meta[j];
        if (j == i || !(mj & kInD)) continue;
        if ((static_cast<uint32_t>(w.top[j]) >> (16 - plen)) != prefix) continue;
        const int32_t yj = entry_y(w, t2, j);
        const uint32_t loj = lo_of(t2, mj, yj), hij = hi_of(t2, mj, yj);
        const uint64_t kj = own_key(kc, t, loj, hij);
        r += (kj < ki || (kj == ki && tie_break(loj, hij) < tbi));
      }
      if (r == kk - 1) {
        out->key = ki;
        out->tb = tbi;
      }
    }
  }
  tm.sync();
  if (cnt > 1 && cnt <= kCand) {
    for (int q = tm.rank; q < cnt; q += Team::N) {
      int r = 0;
      for (int j = 0; j < cnt; ++j) r += (ck[j] < ck[q] || (ck[j] == ck[q] && ctb[j] < ctb[q]));
      if (r == kk - 1) {
        out->key = ck[q];
        out->tb = ctb[q];
      }
    }
    tm.sync();
  }
}

// Trade t (nodes at t2u, t2u+1) depends on the earlier trade s through a
// block of two or more edges (flags f: bit 2 rho + gamma, t's node rho
// adjacent to s's node 2s + gamma): replay s's decisions on the block from
// its published threshold and return whether t's other node is adjacent to
// the s-node that the row-r entry of column colb ends on when t acts (a
// common neighbour).  Kept out of line: the path is rare, and inlined into
// every unrolled entry it would copy Philox many times over.
__device__ __noinline__ int replay_other(const uint64_t* thr_key, const uint64_t* thr_tb, KeyCtx kc, uint32_t t2u,
                                         uint32_t s, uint32_t f, int r, int colb) {
  const int u0 = f & 1, u1 = (f >> 1) & 1, v0 = (f >> 2) & 1, v1 = (f >> 3) & 1;
  const int bits[2][2] = {{u0, u1}, {v0, v1}};
  const int cnt_row[2] = {u0 + u1, v0 + v1};
  int m1[2][2] = {{0, 0}, {0, 0}};
  int col_now = colb;
  const uint64_t tk = __ldcg(thr_key + s), tt = __ldcg(thr_tb + s);
  for (int rho = 0; rho < 2; ++rho)
    for (int gam = 0; gam < 2; ++gam) {
      if (!bits[rho][gam]) continue;
      int g2 = gam;
      if (cnt_row[rho] == 1) {
        const uint32_t x = t2u + rho, yb = 2u * s + gam;
        const uint32_t lo = min(x, yb), hi = max(x, yb);
        const uint64_t k = side_key(kc, lo, hi, (lo >> 1) == s);
        g2 = at_or_below(k, tie_break(lo, hi), tk, tt) ? 0 : 1;
      }
      m1[rho][g2] = 1;
      if (rho == r && gam == colb) col_now = g2;
    }
  return m1[1 - r][col_now];
}

// Phase A for trade t.
// The next trade's bulk copy, issued by member 0 as soon as the current trade
// has read its staged entries (the same buffer is reused).
struct StageNext {
  bool issue;
  int64_t b0;
  int L;
  int32_t* buf;
  uint64_t* mbar;
};

// An unpublished dependency s < wait_below is waited for; any other makes the
// result false (in every member).
template <class Team, bool kOneSeed = false>
__device__ bool phase_a(Team& tm, const StepCtx& c, int64_t t, const WsA& w, SelOut* sel,
                        const int32_t* ystage = nullptr, StageNext sn = StageNext{false, 0, 0, nullptr, nullptr},
                        uint32_t wait_below = 0) {
  const TradeRows tr = trade_rows(c, t);
  const KeyCtx kc = key_ctx<kOneSeed>(c, t);
  const int du = tr.du, dv = tr.dv, L = du + dv;
  const int H = 1 << w.lgH;
  const int64_t t2 = 2 * t;
  for (int i = tm.rank; i < H; i += Team::N) w.hkey[i] = 0u;
  for (int i = tm.rank; i < ((H + 15) & ~15) / 4; i += Team::N) reinterpret_cast<uint32_t*>(w.hflag)[i] = 0u;
  for (int i = tm.rank; i < kSelBins; i += Team::N) w.hist[i] = 0;
  if (tm.rank == 0) *w.ncand = 0;
  tm.sync();
  // entries into the hash: the far trade's slot (open addressing, far trade
  // + 1 as key: a plain store into an empty home slot, read back after a
  // barrier; an entry whose home slot another key won claims a further slot
  // with a compare-and-swap), then the presence bit (row, column) in the
  // slot's flags.  All passes take kBatch entries of a member at a time, loads
  // first: parts of the work space may be in global memory.
  constexpr int N = Team::N, kBatch = 4;
  const uint32_t hmask = (1u << w.lgH) - 1u;
  auto entry = [&](int i) { return ystage ? ystage[i] : __ldcg(c.col + tr.b0 + i); };
  for (int i0 = tm.rank; i0 < L; i0 += N * kBatch) {
    int32_t yy[kBatch];
#pragma unroll
    for (int q = 0; q < kBatch; ++q) yy[q] = i0 + q * N < L ? entry(i0 + q * N) : 0;
#pragma unroll
    for (int q = 0; q < kBatch; ++q) {
      const int i = i0 + q * N;
      if (i >= L) break;
      const int r = i >= du;
      const int64_t s = yy[q] >> 1;
      uint8_t m = static_cast<uint8_t>(r | ((yy[q] & 1) ? kCol : 0));
      int32_t sl = -1;
      if (s == t) {
        m |= kUV;
      } else {
        sl = static_cast<int32_t>(hslot(static_cast<uint32_t>(s), w.lgH));
        if (w.hkey[sl] == 0u) w.hkey[sl] = static_cast<uint32_t>(s) + 1u;
      }
      w.slot[i] = sl;
      w.meta[i] = m;
    }
  }
  tm.sync();
  for (int i0 = tm.rank; i0 < L; i0 += N * kBatch) {
    uint32_t key[kBatch], col[kBatch], at[kBatch], won[kBatch];
#pragma unroll
    for (int q = 0; q < kBatch; ++q) {
      const int i = i0 + q * N;
      const uint32_t yy = i < L ? static_cast<uint32_t>(entry(i)) : 2u * static_cast<uint32_t>(t);
      key[q] = (yy >> 1) + 1u;
      col[q] = yy & 1u;
    }
#pragma unroll
    for (int q = 0; q < kBatch; ++q) {
      at[q] = hslot(key[q] - 1u, w.lgH);
      won[q] = key[q] == static_cast<uint32_t>(t) + 1u ? key[q] : w.hkey[at[q]];   // the edge {u, v} has no slot
    }
#pragma unroll
    for (int q = 0; q < kBatch; ++q) {
      const int i = i0 + q * N;
      if (i >= L || key[q] == static_cast<uint32_t>(t) + 1u) continue;
      uint32_t sl = at[q];
      if (won[q] != key[q]) {   // lost the slot to another key: claim one further on
        sl = h_claim(w.hkey, hmask, key[q], (sl + 1u) & hmask);
        w.slot[i] = static_cast<int32_t>(sl);
      }
      flag_or(w.hflag, static_cast<int>(sl), 1u << (2 * (i >= du ? 1 : 0) + col[q]));
    }
  }
  tm.sync();
  if (sn.issue && tm.rank == 0) stage_issue(c.col, sn.b0, sn.L, sn.buf, sn.mbar);
  // trade and position indices fit 32 bits (n < 2^31)
  const uint32_t t32 = static_cast<uint32_t>(t), T32 = static_cast<uint32_t>(c.T);
  const uint32_t t2u = 2u * t32;
  const uint32_t pu = static_cast<uint32_t>(c.pos_next[c.order[t2]]);
  const uint32_t pv = tr.single ? 0u : static_cast<uint32_t>(c.pos_next[c.order[t2 + 1]]);
  bool defer = false, has_dependents = false;
  int cnt_a = 0;
  // both trades' keys of every edge; entries of blocks of several edges are
  // for the second loop
  for (int i0 = tm.rank; i0 < L; i0 += N * kBatch) {
    int32_t sl[kBatch];
    uint8_t mq[kBatch];
#pragma unroll
    for (int q = 0; q < kBatch; ++q) {
      const int i = i0 + q * N;
      mq[q] = i < L ? w.meta[i] : kUV;
      sl[q] = i < L ? w.slot[i] : -1;
    }
#pragma unroll
    for (int q = 0; q < kBatch; ++q) {
      const int i = i0 + q * N;
      if (i >= L) break;
      uint8_t m = mq[q];
      if (m & kUV) {
        w.far[i] = 0;
        w.top[i] = 0;
        continue;
      }
      const int r = m & kR;
      const uint32_t colb = (m & kCol) ? 1u : 0u;
      const uint32_t s = w.hkey[sl[q]] - 1u;
      const uint32_t f = w.hflag[sl[q]] & 15u;
      const uint32_t x = t2u + r, y = 2u * s + colb;
      const EdgeKeys ek = edge_keys<kOneSeed>(c, kc, min(x, y), max(x, y));
      const bool lo_mine = x < y;
      const uint32_t top = static_cast<uint32_t>((lo_mine ? ek.lo_side : ek.hi_side) >> 48);
      w.top[i] = static_cast<uint16_t>(top);
      w.far[i] = static_cast<uint16_t>((lo_mine ? ek.hi_side : ek.lo_side) >> (64 - kFarBits));
      if (f & (f - 1u)) {
        m |= kPend;
      } else if (!tr.single) {
        m |= kInD;
        cnt_a += (r == 0);
        atomicAdd(&w.hist[top >> (16 - kSelBits)], 1u);
      }
      w.meta[i] = m;
    }
  }
  // blocks of two or more edges: common neighbours and dependencies
  for (int i = tm.rank; i < L; i += Team::N) {
    uint8_t m = w.meta[i];
    if (!(m & kPend)) continue;
    m &= ~kPend;
    const int r = m & kR;
    const int colb = (m & kCol) ? 1 : 0;
    const int sl = w.slot[i];
    const uint32_t s = w.hkey[sl] - 1u;
    const uint32_t f = w.hflag[sl] & 15u;
    const int u0 = f & 1, u1 = (f >> 1) & 1, v0 = (f >> 2) & 1, v1 = (f >> 3) & 1;
    const int cu = u0 + u1, cv = v0 + v1;
    // a later trade s depends on t when one of its own nodes holds exactly
    // one of the block's edges
    if (!tr.single && s > t32 && s < T32 && (u0 + v0 == 1 || u1 + v1 == 1)) has_dependents = true;
    int other = r ? (colb ? u1 : u0) : (colb ? v1 : v0);   // the other row is adjacent when t acts
    if (!tr.single && s < t32 && (cu == 1 || cv == 1)) {
      if (ld_acquire(c.done + s) != kc.g + 1u &&
          !(s < wait_below && wait_published(c.done + s, c.err, kc.g + 1u, c.wait_ns))) {
        defer = true;
        w.meta[i] = m;
        continue;
      }
      other = replay_other(c.thr_key, c.thr_tb, kc, t2u, s, f, r, colb);
    }
    if (!other && !tr.single) {
      m |= kInD;
      cnt_a += (r == 0);
      atomicAdd(&w.hist[static_cast<uint32_t>(w.top[i]) >> (16 - kSelBits)], 1u);
    }
    w.meta[i] = m;
  }
  // one reduction: |A_{u-v}|, any deferral, any later dependent trade
  const int64_t tot = tm.sum(static_cast<int64_t>(cnt_a) | (static_cast<int64_t>(defer) << 32) |
                             (static_cast<int64_t>(has_dependents) << 48));
  if ((tot >> 32) & 0xffff) {
    tm.sync();
    return false;
  }
  const int a = static_cast<int>(tot & 0xffffffff);
  const bool publish_fence = (tot >> 48) != 0;
  const bool no_thr = tr.single || a == 0;   // u keeps nothing of D
  // the bin of the top kSelBits key bits that holds the a-th smallest element
  int bin = 0, cnt = 0, below = 0;
  if (!no_thr) {
    constexpr int bpm = (kSelBins + Team::N - 1) / Team::N;
    const int b0 = tm.rank * bpm;
    int local = 0;
#pragma unroll
    for (int j = 0; j < bpm; ++j)
      if (b0 + j < kSelBins) local += static_cast<int>(w.hist[b0 + j]);
    int run = static_cast<int>(tm.exscan(local));
#pragma unroll
    for (int j = 0; j < bpm; ++j) {
      const int b = b0 + j;
      if (b < kSelBins) {
        const int hc = static_cast<int>(w.hist[b]);
        if (run < a && a <= run + hc) {
          sel->bin = b;
          sel->below = run;
          sel->cnt = hc;
        }
        run += hc;
      }
    }
    tm.sync();
    bin = sel->bin;
    below = sel->below;
    cnt = sel->cnt;
  }
  uint64_t tk = 0, tt = 0;
  if (cnt <= kCand) {
    // the threshold first, so that dependent trades go on: the elements of its
    // bin (the only one, or ranked by full key)
    for (int i0 = tm.rank; cnt > 0 && i0 < L; i0 += N * kBatch) {
      uint32_t mine = 0;
#pragma unroll
      for (int q = 0; q < kBatch; ++q) {
        const int i = i0 + q * N;
        if (i < L && (w.meta[i] & kInD) && (static_cast<int>(w.top[i]) >> (16 - kSelBits)) == bin) mine |= 1u << q;
      }
      for (; mine; mine &= mine - 1u) {
        const int i = i0 + (__ffs(mine) - 1) * N;
        const uint8_t m = w.meta[i];
        const int32_t y = entry_y(w, t2, i);
        const uint32_t lo = lo_of(t2, m, y), hi = hi_of(t2, m, y);
        const int q = cnt == 1 ? 0 : atomicAdd(w.ncand, 1);
        w.ck[q] = own_key(kc, t, lo, hi);
        w.ctb[q] = tie_break(lo, hi);
        w.cidx[q] = i;
      }
    }
    tm.sync();
    const int kk = a - below;
    for (int q = tm.rank; q < cnt; q += Team::N) {
      int rk = 0;
      for (int j = 0; j < cnt; ++j) rk += (w.ck[j] < w.ck[q] || (w.ck[j] == w.ck[q] && w.ctb[j] < w.ctb[q]));
      if (rk == kk - 1) {
        sel->key = w.ck[q];
        sel->tb = w.ctb[q];
      }
      const int i = w.cidx[q];
      const uint8_t m = w.meta[i];
      const int r = m & kR;
      if ((rk < kk ? 0 : 1) != r) {
        w.meta[i] = m | kFlip;
        flag_or(w.hflag, w.slot[i], 16u << (2 * r + ((m & kCol) ? 1 : 0)));
      }
    }
    tm.sync();
    if (!no_thr) {
      tk = sel->key;
      tt = sel->tb;
    }
    if (tm.rank == 0) publish(c, kc, t, pu, pv, tk, tt, publish_fence);
    // own decisions: an element below the threshold's bin stays with u, above
    // it goes to v
    for (int i0 = tm.rank; i0 < L; i0 += N * kBatch) {
      uint8_t mq[kBatch];
      int d[kBatch];
      int32_t sl[kBatch];
#pragma unroll
      for (int q = 0; q < kBatch; ++q) {
        const int i = i0 + q * N;
        mq[q] = i < L ? w.meta[i] : 0;
        d[q] = i < L ? static_cast<int>(w.top[i]) >> (16 - kSelBits) : 0;
        sl[q] = i < L ? w.slot[i] : 0;
      }
#pragma unroll
      for (int q = 0; q < kBatch; ++q) {
        const uint8_t m = mq[q];
        const int r = m & kR;
        if (!(m & kInD) || (!no_thr && d[q] == bin) || (no_thr || d[q] > bin ? 1 : 0) == r) continue;
        w.meta[i0 + q * N] = m | kFlip;
        flag_or(w.hflag, sl[q], 16u << (2 * r + ((m & kCol) ? 1 : 0)));
      }
    }
    tm.sync();
  } else {
    // crowded bin (|D| in the tens of thousands): the general selection
    select_kth(tm, kc, w, L, t, a, sel);
    tk = sel->key;
    tt = sel->tb;
    if (tm.rank == 0) publish(c, kc, t, pu, pv, tk, tt, publish_fence);
    const uint32_t tk16 = static_cast<uint32_t>(tk >> 48);
    for (int i = tm.rank; i < L; i += Team::N) {
      const uint8_t m = w.meta[i];
      if (!(m & kInD)) continue;
      const int r = m & kR;
      const uint32_t tp = w.top[i];
      bool low;
      if (tp != tk16) {
        low = tp < tk16;
      } else {
        const int32_t y = entry_y(w, t2, i);
        const uint32_t lo = lo_of(t2, m, y), hi = hi_of(t2, m, y);
        low = at_or_below(own_key(kc, t, lo, hi), tie_break(lo, hi), tk, tt);
      }
      if ((low ? 0 : 1) != r) {
        w.meta[i] = m | kFlip;
        flag_or(w.hflag, w.slot[i], 16u << (2 * r + ((m & kCol) ? 1 : 0)));
      }
    }
    tm.sync();
  }
  // placement: each entry goes into the new row of its node after the trade
  // (u's or v's row of step g+1) at a slot given by a scan over the team
  int n0 = 0, n1 = 0;
  for (int i = tm.rank; i < L; i += Team::N) {
    const uint8_t m = w.meta[i];
    const int side = (m & kR) ^ ((m & kFlip) ? 1 : 0);
    n0 += side == 0;
    n1 += side;
  }
  const int64_t pre = tm.exscan(static_cast<int64_t>(n0) | (static_cast<int64_t>(n1) << 32));
  int s0 = static_cast<int>(pre & 0xffffffff), s1 = static_cast<int>(pre >> 32);
  if (tm.rank == Team::N - 1 && (s0 + n0 != du || s1 + n1 != dv)) latch(c.err, kErrRowLength);
  const int64_t ou = c.rp_next[pu];
  const int64_t ov = tr.single ? 0 : c.rp_next[pv];
  for (int i0 = tm.rank; i0 < L; i0 += N * kBatch) {
    uint8_t mq[kBatch];
    int32_t slq[kBatch];
    uint16_t far[kBatch];
    uint32_t sq[kBatch], flq[kBatch];
#pragma unroll
    for (int q = 0; q < kBatch; ++q) {
      const int i = i0 + q * N;
      mq[q] = i < L ? w.meta[i] : kUV;
      slq[q] = i < L ? w.slot[i] : -1;
      far[q] = i < L ? w.far[i] : 0;
    }
#pragma unroll
    for (int q = 0; q < kBatch; ++q) {
      const bool uv = (mq[q] & kUV) != 0;
      sq[q] = uv ? 0u : w.hkey[slq[q]] - 1u;
      flq[q] = uv ? 0u : w.hflag[slq[q]];
    }
#pragma unroll
    for (int q = 0; q < kBatch; ++q) {
      if (i0 + q * N >= L) break;
      const uint8_t m = mq[q];
      const int f = (m & kFlip) ? 1 : 0, r = m & kR;
      const uint32_t s = sq[q], fl = flq[q];
      int in_far = 0;
      if (!(m & kUV)) {   // will the far trade decide this edge?
        const int u0 = fl & 1, u1 = (fl >> 1) & 1, v0 = (fl >> 2) & 1, v1 = (fl >> 3) & 1;
        const int cr = r ? (v0 + v1) : (u0 + u1);
        if (tr.single || s < t32) {
          in_far = (cr == 1);                 // trade s acted before t: initial block
        } else if (s < T32) {
          if (u0 + u1 + v0 + v1 == 1) {
            in_far = 1;
          } else {                            // block after t's own decisions: presence bits 0..3, flips 4..7
            const int myrow = r ^ f;
            int same = 0;
#pragma unroll
            for (int b = 0; b < 4; ++b) {
              if (!((fl >> b) & 1)) continue;
              same += (((b >> 1) ^ ((fl >> (4 + b)) & 1)) == myrow);
            }
            in_far = (same == 1);
          }
        }
      }
      const int side = r ^ f;
      const int k = side ? s1++ : s0++;
      if (k >= (side ? dv : du)) continue;   // counts checked above: never write outside the row
      const int64_t slot = (side ? ov : ou) + k;
      c.ph[slot] = m & kUV ? static_cast<int32_t>(t2 + 1 - r) : static_cast<int32_t>(2 * s + ((m & kCol) ? 1 : 0));
      c.fb[slot] = static_cast<uint16_t>(f | (in_far ? ((static_cast<uint32_t>(far[q]) << 1) | kFbInFar) : 0u));
    }
  }
  tm.sync();
  return true;
}

// ------------------------------------------------ register-resident phase A
//
// The same decisions as phase_a for a trade whose L = deg u + deg v entries
// fit the team's registers (J entries per member, entry i held by member
// i mod N): each member keeps its entries' neighbour positions, key bits and
// flags in registers across the passes, so the only shared-memory traffic is
// the far-trade hash, one histogram and the few candidates of the threshold's
// bin.

// Per entry a member keeps the neighbour position y, the top 32 bits of its
// own key, and a word of the far trade's hash slot (bits 0..14) and the far
// key's top kFarBits bits (from bit kMFarShift); per member, one bit per entry
// j for what the entry is (valid, the edge {u, v}, in D, moved, in a
// multi-edge block).
constexpr uint32_t kMSlot = 0x7FFFu;
constexpr int kMFarShift = 21;

// a[j] for a j known at run time (a select chain: a stays in registers)
template <int J>
__device__ __forceinline__ uint32_t pick(const uint32_t (&a)[J], int j) {
  uint32_t v = a[0];
#pragma unroll
  for (int k = 1; k < J; ++k) v = j == k ? a[k] : v;
  return v;
}

__host__ __device__ constexpr int lg_ceil(int x) {
  int lg = 0;
  while ((1 << lg) < x) ++lg;
  return lg;
}

// One team's workspace: a base address and a compile-time layout for trades
// of at most LMAX entries and 2^B histogram bins (four per member).
//
// The far-trade hash has two tables of (key, block word) pairs.  Table 1
// (kH slots, SLOTS per entry) is never cleared: in one round every entry
// stores its key and a zero block word into its home slot, whatever is there,
// so after a barrier each home slot holds a key of this trade.  Only the
// entries that find another key there (about 8 % at 4 to 8 slots per entry)
// go to table 2 (kH2 >= LMAX slots, cleared per trade), by compare-and-swap.
// Clearing the single 8-byte-per-slot table this replaces took 16 stores per
// member; table 2 and the histogram take 3.
template <int LMAX, int B, int CAND, int SLOTS = 4>
struct RegWs {
  static_assert(B >= 5, "tables are cleared in 16-byte stores");
  static constexpr int kLmax = LMAX;
  static constexpr int kCandCap = CAND;                 // candidates ranked directly
  static constexpr int kH = 1 << lg_ceil(SLOTS * LMAX);
  static constexpr int kH2 = 1 << lg_ceil(LMAX);
  static_assert(kH + kH2 <= int(kMSlot) + 1, "slot field");
  static constexpr size_t kCk = 0;                              // candidate keys
  static constexpr size_t kCtb = kCk + CAND * 8;                // candidate tie-breaks
  static constexpr size_t kSel = kCtb + CAND * 8;               // selection results shared by the team
  static constexpr size_t kPw = kSel + ((sizeof(SelOut) + 15) & ~size_t(15));   // radix prefix (4 words)
  static constexpr size_t kNc = kPw + 16;                       // candidate count
  static constexpr size_t kHist = kNc + 16;                     // radix histogram
  static constexpr size_t kHk = kHist + (size_t(1) << B) * 4;   // slots: table 1, then table 2
  static constexpr size_t kBytes = (kHk + size_t(kH + kH2) * 8 + 15) & ~size_t(15);
  static_assert(kHk % 16 == 0 && kHist % 16 == 0, "16-byte aligned tables");
  char* base;
  __device__ __forceinline__ uint64_t* ck() const { return reinterpret_cast<uint64_t*>(base + kCk); }
  __device__ __forceinline__ uint64_t* ctb() const { return reinterpret_cast<uint64_t*>(base + kCtb); }
  __device__ __forceinline__ SelOut* sel() const { return reinterpret_cast<SelOut*>(base + kSel); }
  __device__ __forceinline__ uint32_t* pw() const { return reinterpret_cast<uint32_t*>(base + kPw); }
  __device__ __forceinline__ int32_t* ncand() const { return reinterpret_cast<int32_t*>(base + kNc); }
  __device__ __forceinline__ uint32_t* hist() const { return reinterpret_cast<uint32_t*>(base + kHist); }
  __device__ __forceinline__ uint2* hs() const { return reinterpret_cast<uint2*>(base + kHk); }
};

// Slot of key (far trade + 1) in table 2 (mask + 1 slots at tab, more than
// the keys it can get), starting the probe at p.
__device__ __forceinline__ uint32_t h_claim2(uint2* tab, uint32_t mask, uint32_t key, uint32_t p) {
  for (;;) {
    const uint32_t cur = atomicCAS(&tab[p].x, 0u, key);
    if (cur == 0u || cur == key) return p;
    p = (p + 1u) & mask;
  }
}

// A slot's block word holds one byte per edge of the 2x2 block matrix
// (byte 2 rho + gamma: the trade's node rho adjacent to the far node
// 2s + gamma): 0 absent, 1 present, 3 present and moved by the trade.
// Plain byte stores fill it (the entries of one slot write different bytes,
// or equal values), so it needs no atomics.  block_flags turns it into the
// flag layout of the shared-memory path: presence bits 0..3, flips 4..7.
__device__ __forceinline__ uint32_t compact_bytes(uint32_t x) {   // x: bytes 0 or 1
  return (x | (x >> 7) | (x >> 14) | (x >> 21)) & 15u;
}
__device__ __forceinline__ uint32_t block_flags(uint32_t w) {
  return compact_bytes(w & 0x01010101u) | (compact_bytes((w >> 1) & 0x01010101u) << 4);
}
__device__ __forceinline__ void block_mark(uint2* hs, uint32_t slot, uint32_t q, uint8_t v) {
  reinterpret_cast<uint8_t*>(&hs[slot].y)[q] = v;
}

// Word d of an element's 128-bit order (key, lo, hi): key high, key low, lo, hi.
__device__ __forceinline__ uint32_t sel_word(int d, uint64_t key, uint32_t lo, uint32_t hi) {
  return d == 0 ? static_cast<uint32_t>(key >> 32) : d == 1 ? static_cast<uint32_t>(key) : d == 2 ? lo : hi;
}
// B bits of the 128-bit order starting q bits below its top.
__device__ __forceinline__ uint32_t sel_digit(int q, int B, uint64_t key, uint32_t lo, uint32_t hi) {
  const int w = q >> 5, off = q & 31;
  const uint64_t x = (static_cast<uint64_t>(sel_word(w, key, lo, hi)) << 32) |
                     (w < 3 ? sel_word(w + 1, key, lo, hi) : 0u);
  return static_cast<uint32_t>((x << off) >> (64 - B));
}
// Do the top q bits of the element's order equal those of the prefix pw?
__device__ __forceinline__ bool sel_match(int q, const uint32_t* pw, uint64_t key, uint32_t lo, uint32_t hi) {
  for (int d = 0; d < 4 && 32 * d < q; ++d) {
    const uint32_t a = sel_word(d, key, lo, hi), b = pw[d];
    const int bits = min(32, q - 32 * d);
    if (bits == 32 ? a != b : (a >> (32 - bits)) != (b >> (32 - bits))) return false;
  }
  return true;
}

// The common path is straight-line code over the J entries; everything that
// few entries need (blocks of several edges, slots lost to another key, the
// threshold bin's elements) runs in rolled loops over the member's bit masks,
// so it exists once and stays out of the instruction cache's way.  False (in
// every member) when a dependency has not published.
// kWait: an unpublished dependency s < wait_below is waited for; the keys are
// then computed before the wait, not after it.
template <class Team, int J, int B, bool kKeepKey, bool kOneSeed = false, bool kWait = false, class Ws>
__device__ bool phase_a_reg(Team& tm, const StepCtx& c, int64_t t, const Ws& w, bool active = true,
                            uint32_t wait_below = 0) {
  constexpr int N = Team::N;
  constexpr bool kWarp = N <= 32;   // the team is a warp or part of one
  static_assert((J == 4 || J == 8) && (1 << B) == 4 * N, "four histogram bins per member");
  static_assert(N * J == Ws::kLmax && N * J < (1 << 16), "16-bit placement counts");
  constexpr int kLgH = lg_ceil(Ws::kH), kLgH2 = lg_ceil(Ws::kH2);
  const TradeRows tr = trade_rows(c, t);
  const KeyCtx kc = key_ctx<kOneSeed>(c, t);
  const int du = tr.du, L = active ? tr.du + tr.dv : 0;
  // the nodes' positions in step g+1, loaded now so that their dependent
  // loads overlap the trade's work
  const uint32_t pu = static_cast<uint32_t>(c.pos_next[c.order[2 * t]]);
  const uint32_t pv = tr.single ? 0u : static_cast<uint32_t>(c.pos_next[c.order[2 * t + 1]]);
  const uint32_t t32 = static_cast<uint32_t>(t), T32 = static_cast<uint32_t>(c.T);
  const uint32_t t2u = 2u * t32;
  const unsigned lanes = tm.lanes();
  const unsigned below_me = (1u << (threadIdx.x & 31)) - 1u;
  uint2* const hs = w.hs();
  uint2* const hs2 = hs + Ws::kH;
  {
    const uint4 z = make_uint4(0u, 0u, 0u, 0u);
    reinterpret_cast<uint4*>(w.hist())[tm.rank] = z;
    uint4* h4 = reinterpret_cast<uint4*>(hs2);   // kH2 = J N slots of 8 bytes
    static_assert(Ws::kH2 == J * N, "");
#pragma unroll
    for (int q = 0; q < J / 2; ++q) h4[tm.rank + q * N] = z;
    if (tm.rank == 0) *w.ncand() = 0;
  }
  // entries and their home slots: every entry stores its key there
  uint32_t y[J], mt[J], kt[J], kl[kKeepKey ? J : 1];
  uint32_t hashed = 0, uv = 0;   // entries to other trades; the edge {u, v}
#pragma unroll
  for (int j = 0; j < J; ++j) {
    const int i = tm.rank + j * N;
    y[j] = i < L ? static_cast<uint32_t>(__ldcg(c.col + tr.b0 + i)) : 0u;
  }
#pragma unroll
  for (int j = 0; j < J; ++j) {
    const uint32_t s = y[j] >> 1;
    mt[j] = hslot(s, kLgH);
    kt[j] = 0;
    if (kKeepKey) kl[j] = 0;
    if (tm.rank + j * N < L) {
      if (s == t32) uv |= 1u << j;
      else {
        hashed |= 1u << j;
        hs[mt[j]] = make_uint2(s + 1u, 0u);
      }
    }
  }
  uint32_t valid = hashed | uv;
  // bit j: entry j sits in v's row
  uint32_t in_v = 0;
#pragma unroll
  for (int j = 0; j < J; ++j) in_v |= (tm.rank + j * N >= du ? 1u : 0u) << j;
  tm.sync();
  // an entry whose key is in its slot marks its edge in the slot's block
  // word; the others (another key won the slot) take a slot of table 2
  uint32_t lost = 0;
#pragma unroll
  for (int j = 0; j < J; ++j) {
    if (!((hashed >> j) & 1u)) continue;
    const uint32_t q = 2u * ((in_v >> j) & 1u) + (y[j] & 1u);
    if (hs[mt[j]].x == (y[j] >> 1) + 1u) block_mark(hs, mt[j], q, 1);
    else lost |= 1u << j;
  }
  while (lost) {
    const int j = __ffs(lost) - 1;
    lost &= lost - 1u;
    const uint32_t yj = pick(y, j), s = yj >> 1;
    const uint32_t sl = Ws::kH + h_claim2(hs2, Ws::kH2 - 1u, s + 1u, (s * 0x85EBCA6Bu) >> (32 - kLgH2));
#pragma unroll
    for (int k = 0; k < J; ++k) mt[k] = j == k ? sl : mt[k];
    block_mark(hs, sl, 2u * ((in_v >> j) & 1u) + (yj & 1u), 1);
  }
  tm.sync();
  // both trades' keys of every edge (step-start positions)
  auto keys = [&]() {
#pragma unroll
    for (int j = 0; j < J; ++j) {
      if (!((hashed >> j) & 1u)) continue;
      const uint32_t x = t2u + ((in_v >> j) & 1u), yb = y[j];
      const EdgeKeys ek = edge_keys<kOneSeed>(c, kc, min(x, yb), max(x, yb));
      const bool lo_mine = x < yb;
      kt[j] = static_cast<uint32_t>((lo_mine ? ek.lo_side : ek.hi_side) >> 32);
      if (kKeepKey) kl[j] = static_cast<uint32_t>(lo_mine ? ek.lo_side : ek.hi_side);
      mt[j] |= (static_cast<uint32_t>((lo_mine ? ek.hi_side : ek.lo_side) >> 32) >> (32 - kFarBits)) << kMFarShift;
    }
  };
  if (kWait) keys();
  // blocks of two or more edges: common neighbours and dependencies
  // (their row offsets are needed last: into L2 meanwhile, without a register)
  asm volatile("prefetch.global.L2 [%0];" ::"l"(c.rp_next + pu));
  if (!tr.single) asm volatile("prefetch.global.L2 [%0];" ::"l"(c.rp_next + pv));
  constexpr uint32_t kFlDefer = 1u << 24, kFlDep = 1u << 25, kFlMulti = 1u << 26;
  uint32_t flags = 0, multi = 0;
  uint32_t in_d = tr.single ? 0u : hashed;   // elements of D: the other row is not adjacent to the neighbour
#pragma unroll
  for (int j = 0; j < J; ++j) {
    const uint32_t fw = hs[mt[j] & kMSlot].y;
    if (fw & (fw - 1u)) multi |= 1u << j;
  }
  multi &= hashed;
  for (uint32_t left = multi; left;) {
    const int j = __ffs(left) - 1;
    left &= left - 1u;
    flags |= kFlMulti;
    const uint32_t yj = pick(y, j), s = yj >> 1;
    const int r = (in_v >> j) & 1u, colb = yj & 1u;
    const uint32_t f = block_flags(hs[pick(mt, j) & kMSlot].y) & 15u;
    const int u0 = f & 1, u1 = (f >> 1) & 1, v0 = (f >> 2) & 1, v1 = (f >> 3) & 1;
    const int cu = u0 + u1, cv = v0 + v1;
    if (!tr.single && s > t32 && s < T32 && (u0 + v0 == 1 || u1 + v1 == 1)) flags |= kFlDep;
    int other = r ? (colb ? u1 : u0) : (colb ? v1 : v0);   // the other row is adjacent when t acts
    if (!tr.single && s < t32 && (cu == 1 || cv == 1)) {
      if (ld_acquire(c.done + s) != kc.g + 1u &&
          !(kWait && s < wait_below && wait_published(c.done + s, c.err, kc.g + 1u, c.wait_ns))) {
        flags |= kFlDefer;
        break;
      }
      other = replay_other(c.thr_key, c.thr_tb, kc, t2u, s, f, r, colb);
    }
    if (other) in_d &= ~(1u << j);
  }
  if (!kWait) keys();
  // histogram of the first radix digit
#pragma unroll
  for (int j = 0; j < J; ++j)
    if ((in_d >> j) & 1u) atomicAdd(&w.hist()[kt[j] >> (32 - B)], 1u);
  // one reduction: |A_{u-v}|, and whether any member saw a deferral, a later
  // dependent trade, a multi-edge block (a barrier of larger teams, so it
  // also orders the histogram)
  const uint32_t tot = tm.count_or(__popc(in_d & ~in_v), flags);
  const bool deferred = (tot & kFlDefer) != 0;
  if (deferred) active = false;
  if (!tm.warp_any(active)) {
    tm.sync();
    return !deferred;
  }
  if (!active) valid = hashed = in_d = multi = 0;   // teams in lockstep: the others' trades go on
  const uint32_t a = active ? tot & 0xffffffu : 0u;
  const bool publish_fence = (tot & kFlDep) != 0;
  const bool multi_any = (tot & kFlMulti) != 0;
  const bool no_thr = tr.single || a == 0;   // u keeps nothing of D
  // the edge of entry j and its own key
  auto edge_of = [&](int j, uint32_t* lo, uint32_t* hi) -> uint64_t {
    const uint32_t x = t2u + ((in_v >> j) & 1u), yj = pick(y, j);
    *lo = min(x, yj);
    *hi = max(x, yj);
    if constexpr (kKeepKey) return (static_cast<uint64_t>(pick(kt, j)) << 32) | pick(kl, j);
    else return own_key(kc, t, *lo, *hi);
  };
  if (kWarp) tm.sync();
  uint64_t tk = 0, tt = 0;
  if (tm.warp_any(!no_thr)) {
    // the bin of the first digit (top B key bits) that holds the a-th
    // smallest element: four bins per member
    uint32_t bin = 0, below = 0, cnt = 0;
    {
      const uint4 h = reinterpret_cast<const uint4*>(w.hist())[tm.rank];
      const uint32_t c1 = h.x + h.y, c2 = c1 + h.z, c3 = c2 + h.w;
      const uint32_t run = tm.exscan32(c3);
      const uint32_t k = a - run;   // 1-based rank within the member's bins
      const bool found = a > run && k <= c3;
      uint32_t p = 3, pb = c2, pc = h.w;
      if (k <= c2) { p = 2; pb = c1; pc = h.z; }
      if (k <= c1) { p = 1; pb = h.x; pc = h.y; }
      if (k <= h.x) { p = 0; pb = 0; pc = h.x; }
      if (kWarp) {   // at most 128 entries: 8-bit fields
        const uint32_t info = (4u * tm.rank + p) | ((run + pb) << 8) | (pc << 16);
        const int src = __ffs(__ballot_sync(kFull, found) & lanes) - 1;
        const uint32_t got = __shfl_sync(kFull, info, src & 31);
        bin = got & 0xffu;
        below = (got >> 8) & 0xffu;
        cnt = no_thr ? 0u : got >> 16;
      } else {
        if (found) {
          w.sel()->bin = static_cast<int32_t>(4u * tm.rank + p);
          w.sel()->below = static_cast<int32_t>(run + pb);
          w.sel()->cnt = static_cast<int32_t>(pc);
        }
        tm.sync();
        bin = static_cast<uint32_t>(w.sel()->bin);
        below = static_cast<uint32_t>(w.sel()->below);
        cnt = static_cast<uint32_t>(w.sel()->cnt);
      }
    }
    int qbits = B;              // top bits of the order fixed so far
    uint32_t kk = a - below;    // rank sought among the elements sharing them
    const uint32_t cap = min(static_cast<uint32_t>(c.cand_max), static_cast<uint32_t>(Ws::kCandCap));
    if (tm.warp_any(cnt > cap)) {
      // more elements share the prefix than the candidate list holds (or the
      // list is disabled): further B-bit digits of (key, lo, hi)
      tm.sync();
      if (tm.rank == 0) {
        w.pw()[0] = bin << (32 - B);
        w.pw()[1] = w.pw()[2] = w.pw()[3] = 0u;
      }
      while (tm.warp_any(cnt > cap)) {
        const bool need = cnt > cap;
        reinterpret_cast<uint4*>(w.hist())[tm.rank] = make_uint4(0u, 0u, 0u, 0u);
        tm.sync();
        for (uint32_t left = need ? in_d : 0u; left;) {
          const int j = __ffs(left) - 1;
          left &= left - 1u;
          uint32_t lo, hi;
          const uint64_t key = edge_of(j, &lo, &hi);
          if (sel_match(qbits, w.pw(), key, lo, hi)) atomicAdd(&w.hist()[sel_digit(qbits, B, key, lo, hi)], 1u);
        }
        tm.sync();
        const uint4 h = reinterpret_cast<const uint4*>(w.hist())[tm.rank];
        const uint32_t hv[4] = {h.x, h.y, h.z, h.w};
        uint32_t run = tm.exscan32(h.x + h.y + h.z + h.w);
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          if (need && run < kk && kk <= run + hv[q]) {
            w.sel()->bin = 4 * tm.rank + q;
            w.sel()->below = static_cast<int32_t>(run);
            w.sel()->cnt = static_cast<int32_t>(hv[q]);
          }
          run += hv[q];
        }
        tm.sync();
        const uint32_t dig = static_cast<uint32_t>(w.sel()->bin);
        if (need) {
          kk -= static_cast<uint32_t>(w.sel()->below);
          cnt = static_cast<uint32_t>(w.sel()->cnt);
        }
        if (need && tm.rank == 0) {   // append the digit to the prefix (it may straddle two words)
          const int wd = qbits >> 5, off = qbits & 31;
          const uint64_t d64 = static_cast<uint64_t>(dig) << (64 - B - off);
          w.pw()[wd] |= static_cast<uint32_t>(d64 >> 32);
          if (wd < 3) w.pw()[wd + 1] |= static_cast<uint32_t>(d64);
        }
        if (need) qbits += B;
        tm.sync();
      }
    }
    // rank the few elements that share the prefix by their full order
    uint32_t cand = 0;
#pragma unroll
    for (int j = 0; j < J; ++j) cand |= ((kt[j] >> (32 - B)) == bin ? 1u : 0u) << j;
    for (cand = cnt ? cand & in_d : 0u; cand;) {
      const int j = __ffs(cand) - 1;
      cand &= cand - 1u;
      uint32_t lo, hi;
      const uint64_t key = edge_of(j, &lo, &hi);
      if (qbits > B && !sel_match(qbits, w.pw(), key, lo, hi)) continue;
      if (cnt == 1) {
        w.sel()->key = key;
        w.sel()->tb = tie_break(lo, hi);
      } else {
        const int q = atomicAdd(w.ncand(), 1);
        w.ck()[q] = key;
        w.ctb()[q] = tie_break(lo, hi);
      }
    }
    tm.sync();
    if (tm.warp_any(cnt > 1)) {
      for (uint32_t q = tm.rank; cnt > 1 && q < cnt; q += N) {
        uint32_t rk = 0;
        for (uint32_t p = 0; p < cnt; ++p)
          rk += (w.ck()[p] < w.ck()[q] || (w.ck()[p] == w.ck()[q] && w.ctb()[p] < w.ctb()[q]));
        if (rk == kk - 1) {
          w.sel()->key = w.ck()[q];
          w.sel()->tb = w.ctb()[q];
        }
      }
      tm.sync();
    }
    if (!no_thr) {
      tk = w.sel()->key;
      tt = w.sel()->tb;
    }
  }
  if (active && tm.rank == 0) publish(c, kc, t, pu, pv, tk, tt, publish_fence);
  // own decisions: u keeps the elements at or below the threshold
  const uint32_t tk32 = static_cast<uint32_t>(tk >> 32);
  uint32_t above = 0, equal = 0;
#pragma unroll
  for (int j = 0; j < J; ++j) {
    above |= (kt[j] > tk32 ? 1u : 0u) << j;
    equal |= (kt[j] == tk32 ? 1u : 0u) << j;
  }
  if (no_thr) {
    above = (1u << J) - 1u;
  } else {
    for (equal &= in_d; equal;) {   // the threshold itself, and keys that share its top half
      const int j = __ffs(equal) - 1;
      equal &= equal - 1u;
      uint32_t lo, hi;
      const uint64_t key = edge_of(j, &lo, &hi);
      if (!at_or_below(key, tie_break(lo, hi), tk, tt)) above |= 1u << j;
    }
  }
  const uint32_t flip = (above ^ in_v) & in_d;   // elements that change node
  const uint32_t side = in_v ^ flip;             // the row each entry lands in
  if (tm.warp_any(multi_any)) {
    for (uint32_t left = multi & flip; left;) {
      const int j = __ffs(left) - 1;
      left &= left - 1u;
      block_mark(hs, pick(mt, j) & kMSlot, 2u * ((in_v >> j) & 1u) + (pick(y, j) & 1u), 3);
    }
    tm.sync();
  }
  // will the far trade decide the edge?  (A single-edge block: yes, unless
  // the far node is the untraded one of an odd n, trade index T.)
  uint32_t in_far = 0;
#pragma unroll
  for (int j = 0; j < J; ++j) in_far |= ((y[j] >> 1) < T32 ? 1u : 0u) << j;
  in_far &= hashed;
  for (uint32_t left = multi; left;) {
    const int j = __ffs(left) - 1;
    left &= left - 1u;
    const uint32_t fl = block_flags(hs[pick(mt, j) & kMSlot].y), s = pick(y, j) >> 1;
    int same = 0;
    if (tr.single || s < t32) {   // trade s acted before t: initial block
      same = __popc((in_v >> j) & 1u ? (fl & 12u) : (fl & 3u));
    } else if (s < T32) {         // block after t's own decisions: presence bits 0..3, flips 4..7
      const uint32_t row = (side >> j) & 1u;
#pragma unroll
      for (int q = 0; q < 4; ++q)
        if ((fl >> q) & 1) same += (((q >> 1) ^ ((fl >> (4 + q)) & 1)) == row);
    }
    if (same != 1) in_far &= ~(1u << j);
  }
  // placement: each entry goes into the new row of its node after the trade
  // (u's or v's row of step g+1).  Slots follow (entry index j, lane), by
  // ballots, so the stores of one instruction fill two runs.
  uint32_t s0 = 0, s1 = 0;
  if (!kWarp) {
    const uint32_t nv = __reduce_add_sync(kFull, __popc(valid & side));
    const uint32_t nu = __reduce_add_sync(kFull, __popc(valid & ~side));
    const uint32_t pre = tm.warps_before(nu | (nv << 16));
    s0 = pre & 0xffffu;
    s1 = pre >> 16;
  }
  const int64_t ou = c.rp_next[pu];
  const int64_t ov = tr.single ? 0 : c.rp_next[pv];
  int32_t* const ph_u = c.ph + ou;
  int32_t* const ph_v = c.ph + ov;
  uint16_t* const fb_u = c.fb + ou;
  uint16_t* const fb_v = c.fb + ov;
#pragma unroll
  for (int j = 0; j < J; ++j) {
    const bool mine = (valid >> j) & 1u, to_v = (side >> j) & 1u;
    const unsigned b1 = __ballot_sync(kFull, mine && to_v) & lanes;
    const unsigned b0 = __ballot_sync(kFull, mine && !to_v) & lanes;
    const uint32_t k = (to_v ? s1 : s0) + __popc((to_v ? b1 : b0) & below_me);
    s0 += __popc(b0);
    s1 += __popc(b1);
    if (mine && k < static_cast<uint32_t>(to_v ? tr.dv : du)) {   // checked below: never outside the row
      (to_v ? ph_v : ph_u)[k] = static_cast<int32_t>(y[j]);
      (to_v ? fb_v : fb_u)[k] = static_cast<uint16_t>(
          ((flip >> j) & 1u) | ((in_far >> j) & 1u ? (((mt[j] >> kMFarShift) << 1) | kFbInFar) : 0u));
    }
  }
  // the last warp's counts are the rows' lengths
  if (active && tm.rank == N - 1 && (s0 != static_cast<uint32_t>(du) || s1 != static_cast<uint32_t>(tr.dv)))
    latch(c.err, kErrRowLength);
  tm.sync();
  return !deferred;
}

// Phase A of small trades, one warp per trade (L <= 32 J): eight independent
// warps per CTA, each with its own workspace; no CTA barriers.
constexpr int kWarpJ = 4;                       // entries per lane: trades up to 128 entries
constexpr int kWarpB = 7;                       // first radix digit: 128 bins
constexpr int kWarpWarps = 8;                   // warps per CTA
using WarpWs = RegWs<32 * kWarpJ, kWarpB, kCand>;

// The smallest trades (L <= W J, W = 8 or 16) on teams of W lanes: 32 / W
// trades per warp, so the per-trade work (clearing the tables, scans,
// reductions, the threshold search) takes one warp instruction for all of
// them.
template <int W>
struct LaneCfg {
  static constexpr int B = W == 8 ? 5 : 6;   // ~1 first-digit bin per entry
  using Ws = RegWs<W * kWarpJ, B, 8>;   // a crowded bin (8 of the few entries) takes a further digit
  static constexpr int kTeams = 32 * kWarpWarps / W;   // teams per CTA
  static constexpr size_t kSmem = Ws::kBytes * kTeams;
};
// Phase A of larger trades: a CTA of CT threads holds CT / NT teams of NT
// threads (named barriers), each running one trade at a time with kTeamJ
// entries per thread in registers (L <= NT kTeamJ).
constexpr int kTeamJ = 4;
template <int NT, int J = kTeamJ, int SLOTS = 4>
struct TeamCfg {
  static constexpr int B = NT == 64 ? 8 : NT == 128 ? 9 : NT == 256 ? 10 : NT == 512 ? 11 : 12;   // ~1 bin per entry
  using Ws = RegWs<NT * J, B, kCand, SLOTS>;
  static constexpr int kMax = NT * J;
};
// The first pass of a handle of fewer than kFuseMax trades runs classes 0 to 5
// in one kernel, and 6 and 7 in another.  A class's trades are cut into CTA
// rounds (one trade per team), the classes' rounds follow each other, and CTA
// b takes rounds b, b + G, ...: the classes run side by side on different
// CTAs, where a launch per class spends its time on the latency of one round
// each (n=4096, four classes: 53 us -> 18 in one kernel; n=2^17: 153 -> 135).
// Large graphs keep a kernel per class: CTAs of one SM in different classes
// share its instruction cache badly (n=2^20: 848 us per class, 947 together).
// (kFuseMax in cb_internal.cuh.)
struct Rounds {
  int64_t at = 0;   // rounds of the classes so far
  // this CTA's first round of a class of `rounds`
  __device__ __forceinline__ int64_t first(int64_t rounds) {
    const int64_t G = gridDim.x;
    const int64_t i = (static_cast<int64_t>(blockIdx.x) + G - at % G) % G;
    at += rounds;
    return i;
  }
};

template <int W, bool kOneSeed>
__device__ void run_lanes(const StepCtx& c, const ClassList& cl, char* smem, Rounds& rs) {
  using Cfg = LaneCfg<W>;
  const int id = threadIdx.x / W;
  const typename Cfg::Ws w{smem + Cfg::Ws::kBytes * id};
  LaneTeam<W> tm;
  // a warp's teams run in lockstep, so its loop ends when none has a trade
  const int lead = id & ~(32 / W - 1);
  const int64_t step = static_cast<int64_t>(gridDim.x) * Cfg::kTeams;
  for (int64_t q0 = rs.first((cl.len + Cfg::kTeams - 1) / Cfg::kTeams) * Cfg::kTeams + lead; q0 < cl.len; q0 += step) {
    const int64_t q = q0 + (id - lead);
    const bool active = q < cl.len;
    const int64_t t = cl[active ? q : q0];
    if (!phase_a_reg<LaneTeam<W>, kWarpJ, Cfg::B, true, kOneSeed>(tm, c, t, w, active) && tm.rank == 0) defer_trade(c, t);
  }
}
template <bool kOneSeed>
__device__ void run_warps(const StepCtx& c, const ClassList& cl, char* smem, Rounds& rs) {
  const int wid = threadIdx.x >> 5;
  const WarpWs w{smem + WarpWs::kBytes * wid};
  WarpTeam tm;
  const int64_t step = static_cast<int64_t>(gridDim.x) * kWarpWarps;
  for (int64_t q = rs.first((cl.len + kWarpWarps - 1) / kWarpWarps) * kWarpWarps + wid; q < cl.len; q += step)
    if (!phase_a_reg<WarpTeam, kWarpJ, kWarpB, true, kOneSeed>(tm, c, cl[q], w) && tm.rank == 0)
      defer_trade(c, cl[q]);
}
template <int CT, int NT, bool kOneSeed, int J = kTeamJ, int SLOTS = 4>
__device__ void run_teams(const StepCtx& c, const ClassList& cl, char* smem, int64_t* red, Rounds& rs) {
  constexpr int kTeams = CT / NT;
  using Cfg = TeamCfg<NT, J, SLOTS>;
  using Ws = typename Cfg::Ws;
  const int id = threadIdx.x / NT;
  SubTeam<NT> tm(red + id * SubTeam<NT>::kRedSlots, id);
  const Ws w{smem + Ws::kBytes * id};
  const int64_t step = static_cast<int64_t>(gridDim.x) * kTeams;
  for (int64_t q = rs.first((cl.len + kTeams - 1) / kTeams) * kTeams + id; q < cl.len; q += step)
    if (!phase_a_reg<SubTeam<NT>, J, Cfg::B, false, kOneSeed>(tm, c, cl[q], w) && tm.rank == 0)
      defer_trade(c, cl[q]);
}

// Class K alone.  Instruction issue bounds these kernels (55 to 64 % of the
// slots; L1 at 40 %, L2 and DRAM below 25).  Trades of more than 256 entries run
// with eight entries per member on teams of half the size, which halves what a
// trade costs whatever its size (clearing, scans, the threshold search) and its
// barriers; two hash slots per entry keep four CTAs on an SM.  n=2^25, degrees
// [10,10000), ms per step with four and eight: 257 to 512 entries 3.90 and
// 3.65, to 1024 3.74 and 3.14, to 2048 3.56 and 3.05, to 4096 3.65 and 3.13.  On
// lanes and warps eight cost more than they save (class 0 2.98 and 4.24, 1
// 4.38 and 5.79, 2 3.98 and 5.33, 3 4.40 and 4.09 to 4.52): the bins are twice as
// full, and the rolled loops over their elements run in lockstep.
template <int K>
struct ClassCfg {
  static constexpr int kJ = K < 4 ? 4 : 8, kSlots = K < 4 ? 4 : 2;
  static constexpr int kTeam = (32 << K) / kJ;            // threads per trade
  static constexpr int kThreads = K < 7 ? 256 : 512;      // per CTA
  static constexpr int kCtas = 4 * 256 / kThreads;        // per SM
  static constexpr size_t smem() {
    if constexpr (K < 2) return LaneCfg<kTeam>::kSmem;
    else if constexpr (K == 2) return WarpWs::kBytes * kWarpWarps;
    else return TeamCfg<kTeam, kJ, kSlots>::Ws::kBytes * (kThreads / kTeam);
  }
};
template <int K, bool kOneSeed>
__global__ void __launch_bounds__(ClassCfg<K>::kThreads, ClassCfg<K>::kCtas)
    k_phase_a_class(StepCtx c, const int32_t* lists, const int64_t* ctr) {
  after_previous();
  before_next();
  using Cfg = ClassCfg<K>;
  extern __shared__ __align__(16) char smem[];
  __shared__ int64_t red[K < 3 ? 1 : Cfg::kThreads / 16];   // two slots per warp
  Rounds rs;
  const ClassList cl = class_list(c, lists, ctr, K);
  if constexpr (K < 2) run_lanes<Cfg::kTeam, kOneSeed>(c, cl, smem, rs);
  else if constexpr (K == 2) run_warps<kOneSeed>(c, cl, smem, rs);
  else run_teams<Cfg::kThreads, Cfg::kTeam, kOneSeed, Cfg::kJ, Cfg::kSlots>(c, cl, smem, red, rs);
}

// Classes 0 to 5 (without the lane teams or the teams where an option sends
// their trades elsewhere): 256 threads, the longest trades first.
constexpr int kRunLanes = 1, kRunTeams = 2;
constexpr size_t small_smem() {
  size_t m = LaneCfg<8>::kSmem;
  for (size_t x : {LaneCfg<16>::kSmem, WarpWs::kBytes * kWarpWarps, TeamCfg<64>::Ws::kBytes * 4,
                   TeamCfg<128>::Ws::kBytes * 2, TeamCfg<256>::Ws::kBytes})
    m = x > m ? x : m;
  return m;
}
template <bool kOneSeed>
__global__ void __launch_bounds__(256, 4) k_phase_a_small(StepCtx c, const int32_t* lists,
                                                        const int64_t* ctr, int what) {
  after_previous();
  before_next();
  extern __shared__ __align__(16) char smem[];
  __shared__ int64_t red[4 * SubTeam<64>::kRedSlots];
  static_assert(4 * SubTeam<64>::kRedSlots >= SubTeam<256>::kRedSlots && 4 * SubTeam<64>::kRedSlots >= 2 * SubTeam<128>::kRedSlots, "");
  Rounds rs;
  if (what & kRunTeams) {
    run_teams<256, 256, kOneSeed>(c, class_list(c, lists, ctr, 5), smem, red, rs);
    __syncthreads();   // the next class lays the shared memory out anew
    run_teams<256, 128, kOneSeed>(c, class_list(c, lists, ctr, 4), smem, red, rs);
    __syncthreads();
    run_teams<256, 64, kOneSeed>(c, class_list(c, lists, ctr, 3), smem, red, rs);
    __syncthreads();
  }
  run_warps<kOneSeed>(c, class_list(c, lists, ctr, 2), smem, rs);
  if (what & kRunLanes) {
    __syncthreads();
    run_lanes<16, kOneSeed>(c, class_list(c, lists, ctr, 1), smem, rs);
    __syncthreads();
    run_lanes<8, kOneSeed>(c, class_list(c, lists, ctr, 0), smem, rs);
  }
}

// Classes 7 and 6: 1024 threads.
constexpr size_t kLargeSmem = 2 * TeamCfg<512>::Ws::kBytes > TeamCfg<kBigThreads>::Ws::kBytes
                                  ? 2 * TeamCfg<512>::Ws::kBytes : TeamCfg<kBigThreads>::Ws::kBytes;
template <bool kOneSeed>
__global__ void __launch_bounds__(kBigThreads, 1) k_phase_a_large(StepCtx c, const int32_t* lists,
                                                                const int64_t* ctr) {
  after_previous();
  before_next();
  extern __shared__ __align__(16) char smem[];
  __shared__ int64_t red[SubTeam<kBigThreads>::kRedSlots];
  Rounds rs;
  run_teams<kBigThreads, kBigThreads, kOneSeed>(c, class_list(c, lists, ctr, 7), smem, red, rs);
  __syncthreads();
  run_teams<kBigThreads, 512, kOneSeed>(c, class_list(c, lists, ctr, 6), smem, red, rs);
}

// ------------------------------------------------------ rebuild: fix-up
//
// Phase A leaves every entry in its new row (step g+1 layout) as a
// placeholder: the far end's step-g position y, and a side word (bit 0 the
// own trade's flip, bits 1..kFarBits the top bits of the far trade's key for
// the edge, bit 12 set when the far trade decides the edge).  The fix-up
// replaces each placeholder by the step-(g+1) position of the far end: y
// itself, or the node of y's trade that the trade's threshold gives it.  One
// 8-byte record per far trade holds both of its nodes' new positions and its
// threshold's top 8 bits; the pass runs once per slice of far trades small
// enough for the records to stay in L2, each pass reading every placeholder
// and writing the entries of its slice.  Equal 8-bit prefixes (1 in 256)
// fetch the far threshold's longer prefix; a tie there too (1 in 2^kFarBits)
// needs the full key, hence the edge's own end at the start of the step: the
// node of the entry's row (found by a search of the chunk's row offsets)
// before the own flip.

constexpr int kFixThreads = 256;
constexpr int kFixPer = 8;                             // consecutive entries per thread
constexpr int kFixChunk = kFixThreads * kFixPer;       // entries per chunk

struct FarTrade {
  int32_t x, y;    // new positions of nodes 2s and 2s+1
  uint32_t top;    // threshold prefix (8 bits)
};

// The record as loaded: 8 bytes, or 16 for the wide layout.
template <bool kNarrow>
struct FarRaw {
  uint64_t v;
};
template <>
struct FarRaw<false> {
  int4 v;
};
template <bool kNarrow>
__device__ __forceinline__ FarRaw<kNarrow> far_raw(const void* pack, uint32_t s) {
  if constexpr (kNarrow) return {static_cast<const unsigned long long*>(pack)[s]};
  else return {static_cast<const int4*>(pack)[s]};
}
template <bool kNarrow>
__device__ __forceinline__ FarTrade far_decode(const FarRaw<kNarrow>& r) {
  if constexpr (kNarrow) {
    return {static_cast<int32_t>(r.v & 0x0FFFFFFFu), static_cast<int32_t>((r.v >> 28) & 0x0FFFFFFFu),
            static_cast<uint32_t>(r.v >> 56)};
  } else {
    return {r.v.x, r.v.y, static_cast<uint32_t>(r.v.z)};
  }
}

template <bool kNarrow>
__device__ __forceinline__ FarTrade far_trade(const void* pack, uint32_t s) {
  if constexpr (kNarrow) {
    const uint64_t v = static_cast<const unsigned long long*>(pack)[s];
    return {static_cast<int32_t>(v & 0x0FFFFFFFu), static_cast<int32_t>((v >> 28) & 0x0FFFFFFFu),
            static_cast<uint32_t>(v >> 56)};
  } else {
    const int4 v = static_cast<const int4*>(pack)[s];
    return {v.x, v.y, static_cast<uint32_t>(v.z)};
  }
}

// Row (step g+1 position) holding entry e: the last one whose first entry is <= e.
__device__ __forceinline__ int64_t fix_row(const StepCtx& c, int64_t e) {
  const int64_t ch = e / kRowChunk;
  int64_t lo = c.chunk_row[ch], hi = c.chunk_row[ch + 1];
  while (lo < hi) {
    const int64_t mid = (lo + hi + 1) >> 1;
    if (c.rp_next[mid] <= e) lo = mid; else hi = mid - 1;
  }
  return lo;
}

constexpr int kFixQueue = 2 * kFixChunk;    // prefix ties a CTA defers before resolving them together

// The kFixPer placeholders and side words of a thread starting at entry base
// (entries at or past nnz read as 0xFFFFFFFF).
template <bool kStream>
__device__ __forceinline__ void fix_load(const int32_t* ph, const uint16_t* fb, int64_t base, int64_t nnz,
                                         uint32_t* pv, uint32_t* bv) {
  if (base + kFixPer <= nnz) {   // 32 B and 16 B, aligned: chunks start at multiples of 2048 entries
    const uint4* p4 = reinterpret_cast<const uint4*>(ph + base);
    const uint4 a0 = kStream ? __ldcs(p4) : __ldcg(p4);
    const uint4 a1 = kStream ? __ldcs(p4 + 1) : __ldcg(p4 + 1);
    pv[0] = a0.x; pv[1] = a0.y; pv[2] = a0.z; pv[3] = a0.w;
    pv[4] = a1.x; pv[5] = a1.y; pv[6] = a1.z; pv[7] = a1.w;
    const uint4 b = __ldcs(reinterpret_cast<const uint4*>(fb + base));
    bv[0] = b.x; bv[1] = b.y; bv[2] = b.z; bv[3] = b.w;
  } else {
#pragma unroll
    for (int j = 0; j < kFixPer / 2; ++j) bv[j] = 0;
#pragma unroll
    for (int j = 0; j < kFixPer; ++j) {
      const bool in = base + j < nnz;
      pv[j] = in ? static_cast<uint32_t>(ph[base + j]) : 0xFFFFFFFFu;
      if (in) bv[j >> 1] |= static_cast<uint32_t>(fb[base + j]) << (16 * (j & 1));
    }
  }
}

// The new position of entry e's far end when its 8-bit key prefix equals
// the far threshold's: the threshold's longer prefix, and on a tie there too
// the full key of the edge (its own end at the start of the step is the
// node of the entry's row before the own flip).
template <bool kNarrow>
__device__ uint32_t fix_tie(const StepCtx& c, int64_t e, uint32_t y, uint32_t b) {
  const uint32_t s = y >> 1;
  const FarTrade ft = far_trade<kNarrow>(c.far_pack, s);
  const uint32_t fp = (b >> 1) & ((1u << kFarBits) - 1u);
  const uint32_t tp = static_cast<uint32_t>(__ldcg(c.thr_key + s) >> (64 - kFarBits));
  bool low;
  if (fp != tp) {
    low = fp < tp;
  } else {
    const uint32_t xr = static_cast<uint32_t>(c.pos[c.order_next[fix_row(c, e)]]) ^ (b & 1u);
    low = far_keeps_low(c, key_ctx<false>(c, s), s, min(xr, y), max(xr, y));
  }
  return static_cast<uint32_t>(low ? ft.x : ft.y);
}

// The end of a super step, by the last CTA of its last kernel to finish: every
// graph's step counter moves on, the next step's counters are cleared.
struct StepEnd {
  Seg* segs;
  int nseg;
  int64_t* ctr;              // the next step's counters (null: cleared before, as its class lists are built)
  unsigned long long* left;  // CTAs finished (zero between steps)
  int32_t* def_seg;          // deferred trades per segment, cleared
};
__device__ __forceinline__ void end_step(const StepEnd& e) {
  __shared__ int last;
  __syncthreads();
  if (threadIdx.x == 0) {
    __threadfence();
    last = atomicAdd(e.left, 1ull) == gridDim.x - 1;
  }
  __syncthreads();
  if (!last) return;
  for (int i = threadIdx.x; i < e.nseg; i += blockDim.x) e.segs[i].g += 1;
  for (int i = threadIdx.x; e.ctr && i < kCounters; i += blockDim.x) e.ctr[i] = 0;
  for (int i = threadIdx.x; i < kDefKinds * kDefSegs; i += blockDim.x) e.def_seg[i] = 0;
  if (threadIdx.x == 0) *e.left = 0;
}
// ... of a handle without entries.
__global__ void k_step_end(StepEnd e) { end_step(e); }

// One pass over far trades [s_lo, s_hi).  A pass other than the last writes
// the new positions of its entries into the placeholders (marked kPhDone);
// the last one writes every entry's new position to `out` in full vectors.
// Entries whose 8-bit prefix ties wait in a per-CTA queue and are resolved
// together, so that their extra loads hold up no warp.
template <bool kNarrow, bool kLast>
__global__ void __launch_bounds__(kFixThreads, 4) k_fixup(StepCtx c, int64_t nnz, uint32_t s_lo, uint32_t s_hi,
                                                       int32_t* ph, const uint16_t* fb,
                                                       int32_t* out, StepEnd end) {
  after_previous();
  before_next();
  __shared__ int64_t qe[kFixQueue];
  __shared__ int qn;
  if (threadIdx.x == 0) qn = 0;
  __syncthreads();
  auto flush = [&]() {
    const int k = qn;
    for (int i = threadIdx.x; i < k; i += blockDim.x) {
      const int64_t e = qe[i];
      const uint32_t y = static_cast<uint32_t>(ph[e]);
      const uint32_t v = fix_tie<kNarrow>(c, e, y, fb[e]);
      if (kLast) out[e] = static_cast<int32_t>(v);
      else ph[e] = static_cast<int32_t>(v | kPhDone);
    }
    __syncthreads();
    if (threadIdx.x == 0) qn = 0;
    __syncthreads();
  };
  const int64_t nchunks = (nnz + kFixChunk - 1) / kFixChunk;
  const int64_t tofs = static_cast<int64_t>(threadIdx.x) * kFixPer;
  uint32_t pv[kFixPer], bv[kFixPer / 2];
  int64_t ch = blockIdx.x;
  if (ch < nchunks) fix_load<kLast>(ph, fb, ch * kFixChunk + tofs, nnz, pv, bv);
  for (; ch < nchunks; ch += gridDim.x) {
    const int64_t base = ch * kFixChunk + tofs;
    // the next chunk's loads go out before this chunk's gathers
    uint32_t pn[kFixPer], bn[kFixPer / 2];
    const int64_t nxt = ch + gridDim.x;
    if (nxt < nchunks) fix_load<kLast>(ph, fb, nxt * kFixChunk + tofs, nnz, pn, bn);
    // first every gather of the thread's entries in this slice, then the decisions
    bool full = false;   // this thread took a place that leaves no room for a chunk more
    uint32_t res[kFixPer];
    FarRaw<kNarrow> ftv[kFixPer];
    uint32_t todo = 0;   // bit j: entry j is this pass's
#pragma unroll
    for (int j = 0; j < kFixPer; ++j) {
      const uint32_t p = pv[j];
      res[j] = (p & kPhDone) && p != 0xFFFFFFFFu ? (p & ~kPhDone) : 0u;   // an earlier pass resolved it
      const uint32_t s = p >> 1;
      const bool mine = !(p & kPhDone) && s >= s_lo && s < s_hi && p < static_cast<uint32_t>(c.n);
      if (!(p & kPhDone) && p >= static_cast<uint32_t>(c.n)) latch(c.err, kErrRowLength);
      if (mine) ftv[j] = far_raw<kNarrow>(c.far_pack, s);
      todo |= static_cast<uint32_t>(mine) << j;
    }
#pragma unroll
    for (int j = 0; j < kFixPer; ++j) {
      if (!((todo >> j) & 1u)) continue;
      const uint32_t y = pv[j];
      const FarTrade ft = far_decode<kNarrow>(ftv[j]);
      const uint32_t b = (bv[j >> 1] >> (16 * (j & 1))) & 0xFFFFu;
      int side = static_cast<int>(y & 1u);
      if (b & kFbInFar) {   // the far trade decides: key prefixes first
        const uint32_t f8 = ((b >> 1) & ((1u << kFarBits) - 1u)) >> (kFarBits - 8);
        if (f8 == ft.top) {   // 1 in 256: resolved with the queue
          const int at = atomicAdd(&qn, 1);
          qe[at] = base + j;
          full |= at >= kFixQueue - kFixChunk;
          continue;
        }
        side = f8 < ft.top ? 0 : 1;
      }
      res[j] = static_cast<uint32_t>(side ? ft.y : ft.x);
      if (!kLast) ph[base + j] = static_cast<int32_t>(res[j] | kPhDone);
    }
    if (kLast) {
      if (base + kFixPer <= nnz) {
        uint4* o4 = reinterpret_cast<uint4*>(out + base);
        __stcs(o4, make_uint4(res[0], res[1], res[2], res[3]));
        __stcs(o4 + 1, make_uint4(res[4], res[5], res[6], res[7]));
      } else {
#pragma unroll
        for (int j = 0; j < kFixPer; ++j)
          if (base + j < nnz) out[base + j] = static_cast<int32_t>(res[j]);
      }
    }
    // queued entries (and, on the last pass, their vector stores) are in place.
    // The barrier carries the decision to flush: a look at qn after it could
    // see the next chunk's entries of a faster warp, and differ between warps.
    if (__syncthreads_or(full)) flush();
#pragma unroll
    for (int j = 0; j < kFixPer; ++j) pv[j] = pn[j];
#pragma unroll
    for (int j = 0; j < kFixPer / 2; ++j) bv[j] = bn[j];
  }
  __syncthreads();
  flush();
  if (kLast) end_step(end);
}

// ---------------------------------------------------------------- team paths

template <int NT, bool kOneSeed>
__global__ void __launch_bounds__(NT, NT == 256 ? 4 : 1) k_phase_a_block(StepCtx c, const int32_t* lists,
                                                      const int64_t* ctr, int cls, int smem_max,
                                                      size_t room, char* gws, size_t slice, int stage_cap) {
  after_previous();
  before_next();
  // dynamic shared memory: the workspace (room bytes, a multiple of 128), then
  // the staging buffer of a trade's entries (stage_cap + 8 int32)
  extern __shared__ __align__(16) char sbuf[];
  __shared__ int64_t red[BlockTeam<NT>::kRedSlots];
  __shared__ SelOut sel;
  __shared__ uint64_t mbar;
  BlockTeam<NT> tm(red);
  const ClassList cl = class_list(c, lists, ctr, cls);
  const int64_t len = cl.len;
  int32_t* stage = reinterpret_cast<int32_t*>(sbuf + room);
  if (threadIdx.x == 0) {
    mbar_init(&mbar, 1);
    mbar_fence_init();
  }
  __syncthreads();
  uint32_t parity = 0;
  // member 0 reads the next trade's row range at the start of each trade; the
  // copy goes out once the current trade has read its staged entries
  auto range_of = [&](int64_t q, int64_t* b0, int* L) {
    const int64_t t = cl[q];
    const TradeRows tr = trade_rows(c, t);
    *b0 = tr.b0;
    *L = tr.du + tr.dv;
  };
  int64_t nb0 = 0;
  int nL = 0;
  // a trade is staged when it has entries and fits the buffer (every thread
  // applies the same test to the same trade)
  auto staged = [&](int L) { return L > 0 && L <= stage_cap; };
  if (threadIdx.x == 0 && blockIdx.x < len) {
    range_of(blockIdx.x, &nb0, &nL);
    if (staged(nL)) stage_issue(c.col, nb0, nL, stage, &mbar);
  }
  bool failed = false;
  for (int64_t q = blockIdx.x; q < len; q += gridDim.x) {
    const int64_t t = cl[q];
    const TradeRows tr = trade_rows(c, t);
    const int L = tr.du + tr.dv;
    if (L > smem_max && threadIdx.x == 0) atomicAdd(c.gws_count, 1ull);
    const WsA ws = L > smem_max ? carve_split(sbuf, room, gws + slice * blockIdx.x, L) : carve_a(sbuf, L);
    StageNext sn{false, 0, 0, stage, &mbar};
    if (threadIdx.x == 0 && q + gridDim.x < len) {
      range_of(q + gridDim.x, &nb0, &nL);
      sn.issue = staged(nL);
      sn.b0 = nb0;
      sn.L = nL;
    }
    const int32_t* ys = nullptr;
    if (staged(L)) {   // this trade's entries were staged by the previous one (or the prologue)
      const bool late = !mbar_wait(&mbar, parity, c.wait_ns);
      parity ^= 1;
      if (__syncthreads_or(late)) {
        failed = true;
        break;
      }
      ys = stage + stage_off(tr.b0);
    }
    if (!phase_a<BlockTeam<NT>, kOneSeed>(tm, c, t, ws, &sel, ys, sn) && threadIdx.x == 0)
      defer_trade(c, t);
  }
  if (failed) {   // a copy did not complete in time: report, let it land, leave
    if (threadIdx.x == 0) latch(c.err, kErrStage);
    mbar_wait(&mbar, parity ^ 1, c.wait_ns);
  }
}

// A retry pass runs every listed trade once, without waiting; a trade whose
// dependency still has not published is deferred again.  One kernel per list:
// warps claim the small trades one at a time, 256-thread CTAs the medium ones,
// 1024-thread CTAs the large ones.  (One launch with CTAs shared out over the
// lists took 1.06 ms per pass at n=2^25 against 0.6 for two such passes.)
template <int NT>
size_t resolve_smem(int gen_max, int64_t max_trade) {
  const size_t s = std::max(std::max(std::max(TeamCfg<NT>::Ws::kBytes, TeamCfg<256>::Ws::kBytes * (NT / 256)),
                                     ws_a_bytes(std::max(gen_max, 1))),
                            WarpWs::kBytes * (NT / 32));
  return NT == kBigThreads && max_trade > std::min(gen_max, TeamCfg<NT>::kMax) ? std::max(s, kSplitSmem) : s;
}
// A trade of more than kDefMedium entries on the whole CTA.  4097 to 8192
// entries, which the shared-memory form takes three times as long for, fit
// eight to a member of 1024 (two hash slots per entry instead of four: table 2
// takes a fifth of the entries).
using HugeWs = RegWs<8 * kBigThreads, 12, kCand, 2>;
static_assert(HugeWs::kBytes <= kSplitSmem, "");
template <int NT, bool kWait, bool kOneSeed = false>
__device__ bool run_large(BlockTeam<NT>& tm, const StepCtx& c, int64_t t, char* sbuf, SelOut* sel, int gen_max, size_t room,
                          char* gws, size_t slice, uint32_t wait_below) {
  using Ws = typename TeamCfg<NT>::Ws;
  const TradeRows tr = trade_rows(c, t);
  const int L = tr.du + tr.dv;
  if (L <= Ws::kLmax)
    return phase_a_reg<BlockTeam<NT>, kTeamJ, TeamCfg<NT>::B, false, kOneSeed, kWait>(tm, c, t, Ws{sbuf}, true, wait_below);
  if constexpr (NT == kBigThreads)
    if (L <= min(HugeWs::kLmax, gen_max) && HugeWs::kBytes <= room)
      return phase_a_reg<BlockTeam<NT>, 8, 12, false, kOneSeed, kWait>(tm, c, t, HugeWs{sbuf}, true, wait_below);
  if (L > gen_max && threadIdx.x == 0) atomicAdd(c.gws_count, 1ull);
  const WsA ws = L > gen_max ? carve_split(sbuf, room, gws + slice * blockIdx.x, L) : carve_a(sbuf, L);
  return phase_a<BlockTeam<NT>, kOneSeed>(tm, c, t, ws, sel, nullptr, StageNext{false, 0, 0, nullptr, nullptr}, wait_below);
}
// The first pass's largest class: more than min(4096, smem_max) entries, up to
// 8192 of them in registers.  n=2^25, degrees [10,10000): 7.4 ms per step with
// the shared-memory form (k_phase_a_block) up to 8192 entries, 4.7 so.
template <bool kOneSeed>
__global__ void __launch_bounds__(kBigThreads, 1) k_phase_a_huge(StepCtx c, const int32_t* lists,
                                                               const int64_t* ctr, int gen_max,
                                                               char* gws, size_t slice) {
  after_previous();
  before_next();
  extern __shared__ __align__(16) char sbuf[];
  __shared__ int64_t red[BlockTeam<kBigThreads>::kRedSlots];
  __shared__ SelOut sel;
  BlockTeam<kBigThreads> tm(red);
  const ClassList cl = class_list(c, lists, ctr, 8);
  for (int64_t q = blockIdx.x; q < cl.len; q += gridDim.x) {
    const int64_t t = cl[q];
    const TradeRows tr = trade_rows(c, t);
    const int L = tr.du + tr.dv;
    bool ok;
    if (L <= min(HugeWs::kLmax, gen_max)) {
      ok = phase_a_reg<BlockTeam<kBigThreads>, 8, 12, false, kOneSeed>(tm, c, t, HugeWs{sbuf});
    } else {
      if (threadIdx.x == 0) atomicAdd(c.gws_count, 1ull);
      ok = phase_a<BlockTeam<kBigThreads>, kOneSeed>(tm, c, t, carve_split(sbuf, kSplitSmem, gws + slice * blockIdx.x, L),
                                                    &sel);
    }
    if (!ok && threadIdx.x == 0) defer_trade(c, t);
  }
}

__global__ void __launch_bounds__(32 * kWarpWarps, 4) k_retry_warp(StepCtx c, const int32_t* list,
                                                                const unsigned long long* count,
                                                                unsigned long long* claim) {
  extern __shared__ __align__(16) char wsm[];
  const int wid = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const WarpWs w{wsm + WarpWs::kBytes * wid};
  WarpTeam tm;
  const int64_t nl = static_cast<int64_t>(*count);
  for (;;) {
    int64_t p = 0;
    if (lane == 0) p = static_cast<int64_t>(atomicAdd(claim, 1ull));
    p = static_cast<int64_t>(tm.bcast(static_cast<uint64_t>(p), 0));
    if (p >= nl) return;
    if (!phase_a_reg<WarpTeam, kWarpJ, kWarpB, true>(tm, c, list[p], w) && lane == 0) defer_trade(c, list[p]);
  }
}
template <int NT>
__global__ void __launch_bounds__(NT, NT == 256 ? 4 : 1) k_retry(StepCtx c, const int32_t* list,
                                                              const unsigned long long* count,
                                                              unsigned long long* claim, int gen_max, size_t room,
                                                              char* gws, size_t slice) {
  extern __shared__ __align__(16) char sbuf[];
  __shared__ int64_t red[BlockTeam<NT>::kRedSlots];
  __shared__ SelOut sel;
  __shared__ int64_t pick;
  BlockTeam<NT> tm(red);
  const int64_t nl = static_cast<int64_t>(*count);
  for (;;) {
    if (threadIdx.x == 0) pick = static_cast<int64_t>(atomicAdd(claim, 1ull));
    __syncthreads();
    const int64_t p = pick;
    __syncthreads();
    if (p >= nl) return;
    const int32_t t = list[NT == kMedThreads ? -p : p];   // the medium trades' list runs backwards (pair_lists.cuh)
    if (!run_large<NT, false>(tm, c, t, sbuf, &sel, gen_max, room, gws, slice, 0u) && threadIdx.x == 0) defer_trade(c, t);
  }
}

// The in-order pass runs in two kernels.  k_def_list writes the deferred
// trades in index order and cuts the list into chunks of about equal work (a
// large trade, or four medium, or up to 32 small ones).  k_resolve's CTAs
// claim chunks in order; a chunk's small trades run on the CTA's warps, its
// medium ones on teams of 256 threads, its large ones on the whole CTA.  A
// trade waits for an unpublished dependency of an earlier chunk, and is tried
// again when the dependency is in its own.
//
// Every wait ends: every chunk, a CTA's first one too, is claimed from one
// counter in index order, so the chunks before a claimed one are finished or
// held by CTAs that run.  The smallest unfinished trade is then in a claimed
// chunk (or the CTAs come to it), everything its CTA waits for is finished,
// and the CTA comes to it; by induction on the index all trades are run,
// whichever CTAs of the grid are resident.  (A first chunk by block index would
// be held by a CTA that may not have started, while the running ones wait for
// its trades: with other streams' kernels on the SMs it may never start.)
// Chains of dependent trades advance at the pace of the published thresholds.
// A wait that runs out latches kErrResolve; after any error all leave.
constexpr int kChunkWork = 32, kWorkMedium = 8;   // work of a chunk (= a large trade), of a medium trade

// Work of a small and of a medium trade: 1 and 8 when there are many, up to
// a chunk's when that would leave CTAs without a chunk.
__device__ __forceinline__ int chunk_work(int64_t n, int ctas, int least) {
  const int64_t w = n ? int64_t(2 * kChunkWork) * ctas / n : least;
  return static_cast<int>(w < least ? least : w > kChunkWork ? kChunkWork : w);
}

constexpr int kDefListThreads = 256;
__global__ void __launch_bounds__(kDefListThreads) k_def_list(StepCtx c, int64_t nwords, int nsegs, int ctas,
                                                             int32_t* list,
                                                             int32_t* chunk_first,
                                                             unsigned long long* nchunks,
                                                             int64_t* clear) {
  after_previous();
  before_next();
  if (clear && blockIdx.x == 0)   // the next step's counters
    for (int i = threadIdx.x; i < kCounters; i += kDefListThreads) clear[i] = 0;
  __shared__ int64_t red[BlockTeam<kDefListThreads>::kRedSlots];
  const int64_t n0 = static_cast<int64_t>(c.def_n[0]);
  const int64_t total = n0 + static_cast<int64_t>(c.def_n[1] + c.def_n[2]);
  if (total == 0) return;
  BlockTeam<kDefListThreads> tm(red);
  const int work[kDefKinds] = {chunk_work(n0, ctas, 1), chunk_work(static_cast<int64_t>(c.def_n[1]), ctas, kWorkMedium),
                               kChunkWork};
  const int64_t seg_words = c.def_seg_trades / 32;
  for (int seg = blockIdx.x; seg < nsegs; seg += gridDim.x) {
    int mine = 0;
    for (int k = 0; k < kDefKinds; ++k) mine += c.def_seg[k * kDefSegs + seg];
    if (mine == 0) continue;
    // trades and work before this segment
    int64_t before = 0, wbefore = 0;
    for (int i = threadIdx.x; i < seg; i += kDefListThreads)
      for (int k = 0; k < kDefKinds; ++k) {
        const int64_t v = c.def_seg[k * kDefSegs + i];
        before += v;
        wbefore += v * work[k];
      }
    before = tm.sum(before);
    wbefore = tm.sum(wbefore);
    const int64_t w1 = (seg + 1) * seg_words < nwords ? (seg + 1) * seg_words : nwords;
    for (int64_t w0 = seg * seg_words; w0 < w1; w0 += kDefListThreads) {
      const int64_t w = w0 + threadIdx.x;
      const uint32_t bits = w < w1 ? c.def_bits[w] : 0u;
      if (bits) c.def_bits[w] = 0u;   // clear for the next step
      int64_t sum = 0;
      uint64_t kinds = 0;
      int q = 0;
      for (uint32_t left = bits; left; left &= left - 1u, ++q) {
        const TradeRows tr = trade_rows(c, 32 * w + __ffs(left) - 1);
        const int k = def_kind(tr.du + tr.dv);
        kinds |= static_cast<uint64_t>(k) << (2 * q);
        sum += work[k];
      }
      const int64_t mix = (sum << 32) | q;
      const int64_t pre = tm.exscan(mix), all = tm.sum(mix);
      int64_t at = before + (pre & 0xffffffff), wat = wbefore + (pre >> 32);
      for (uint32_t left = bits; left; left &= left - 1u) {
        const int wk = work[kinds & 3u];
        list[at] = static_cast<int32_t>(32 * w + __ffs(left) - 1);
        kinds >>= 2;
        // a trade is in the chunk its work begins in; work is at most
        // kChunkWork, so no chunk number is skipped
        const int64_t ch = wat / kChunkWork;
        if (at == 0) chunk_first[0] = 0;
        ++at;
        wat += wk;
        if (wat / kChunkWork > ch || at == total) chunk_first[ch + 1] = static_cast<int32_t>(at);
        if (at == total) *nchunks = static_cast<unsigned long long>(ch + 1);
      }
      before += all & 0xffffffff;
      wbefore += all >> 32;
    }
  }
}

template <int NT, bool kOneSeed>
__global__ void __launch_bounds__(NT, NT == 256 ? 4 : 1) k_resolve(StepCtx c, const int32_t* list,
                                                                const int32_t* chunk_first,
                                                                const unsigned long long* nchunks,
                                                                unsigned long long* claim, int gen_max, size_t room,
                                                                char* gws, size_t slice) {
  after_previous();
  before_next();
  using Ws256 = typename TeamCfg<256>::Ws;
  constexpr int kWarps = NT / 32, kTeams = NT / 256;
  extern __shared__ __align__(16) char sbuf[];
  __shared__ int64_t red[BlockTeam<NT>::kRedSlots];
  __shared__ int64_t red256[kTeams * SubTeam<256>::kRedSlots];
  __shared__ SelOut sel;
  __shared__ int64_t pick;
  __shared__ int32_t trades[kDefKinds][kChunkWork];   // the chunk's, by kind; -1 once done
  __shared__ int n[kDefKinds], left;
  const int64_t chunks = static_cast<int64_t>(*nchunks);   // 0: nothing was deferred
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, id = threadIdx.x / 256;
  BlockTeam<NT> tm(red);
  SubTeam<256> st(red256 + id * SubTeam<256>::kRedSlots, id);
  WarpTeam wt;
  const WarpWs ww{sbuf + WarpWs::kBytes * warp};
  const Ws256 w256{sbuf + Ws256::kBytes * id};
  if (blockIdx.x >= c.inorder_ctas) return;
  for (;;) {
    // (claimed only now: a chunk held while the one before it waits would hold
    // up others; the first claim and the load of *nchunks go out together)
    if (threadIdx.x == 0) pick = static_cast<int64_t>(atomicAdd(claim, 1ull));
    __syncthreads();
    const int64_t ch = pick;   // written again only after the barriers of this chunk
    if (ch >= chunks) return;
    const int32_t first = chunk_first[ch], count = chunk_first[ch + 1] - first;
    const uint32_t from = static_cast<uint32_t>(list[first]);   // trades before it are in earlier chunks
    if (warp == 0) {
      const int32_t t = lane < count ? list[first + lane] : -1;
      int k = -1;
      if (t >= 0) {
        const TradeRows tr = trade_rows(c, t);
        k = def_kind(tr.du + tr.dv);
      }
#pragma unroll
      for (int q = 0; q < kDefKinds; ++q) {
        const unsigned b = __ballot_sync(kFull, k == q);
        if (k == q) trades[q][__popc(b & ((1u << lane) - 1u))] = t;
        if (lane == 0) n[q] = __popc(b);
      }
    }
    __syncthreads();
    for (;;) {
      if (threadIdx.x == 0) left = 0;
      __syncthreads();
      for (int i = warp; i < n[0]; i += kWarps) {
        const int32_t t = trades[0][i];
        if (t < 0) continue;
        const bool ok = phase_a_reg<WarpTeam, kWarpJ, kWarpB, true, kOneSeed, true>(wt, c, t, ww, true, from);
        if (lane == 0) {
          if (ok) trades[0][i] = -1;
          else atomicAdd(&left, 1);
        }
      }
      if (n[1]) {
        __syncthreads();
        for (int i = id; i < n[1]; i += kTeams) {
          const int32_t t = trades[1][i];
          if (t < 0) continue;
          const bool ok =
              phase_a_reg<SubTeam<256>, kTeamJ, TeamCfg<256>::B, false, kOneSeed, true>(st, c, t, w256, true, from);
          if (st.rank == 0) {
            if (ok) trades[1][i] = -1;
            else atomicAdd(&left, 1);
          }
        }
      }
      for (int i = 0; i < n[2]; ++i) {
        __syncthreads();
        const int32_t t = trades[2][i];
        if (t < 0) continue;
        const bool ok = run_large<NT, true, kOneSeed>(tm, c, t, sbuf, &sel, gen_max, room, gws, slice, from);
        __syncthreads();
        if (threadIdx.x == 0) {
          if (ok) trades[2][i] = -1;
          else atomicAdd(&left, 1);
        }
      }
      __syncthreads();
      const bool more = left != 0;
      if (__syncthreads_or(threadIdx.x == 0 && ld_volatile_i32(c.err) != 0)) return;
      if (!more) break;
    }
  }
}

}  // namespace

namespace {
template <int K>
using Int = std::integral_constant<int, K>;
// Attributes of the kernels built in a one-graph and a general version.
template <bool kOneSeed>
int init_seed_kernels(Graph* h) {
  CB_CUDA(h, cudaFuncSetAttribute(k_phase_a_block<kMedThreads, kOneSeed>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                  static_cast<int>(block_smem_bytes(kBlockMaxCap))));
  CB_CUDA(h, cudaFuncSetAttribute(k_phase_a_block<kBigThreads, kOneSeed>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                  static_cast<int>(std::max(block_smem_bytes(kSmemMaxCap), kSplitSmem))));
  auto of_class = [&](auto k) -> int {
    constexpr int K = decltype(k)::value;
    CB_CUDA(h, cudaFuncSetAttribute(k_phase_a_class<K, kOneSeed>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                    static_cast<int>(ClassCfg<K>::smem())));
    CB_CUDA(h, cudaFuncSetAttribute(k_phase_a_class<K, kOneSeed>, cudaFuncAttributePreferredSharedMemoryCarveout,
                                    cudaSharedmemCarveoutMaxShared));
    return CB_OK;
  };
  int rc;
  if ((rc = of_class(Int<0>{})) || (rc = of_class(Int<1>{})) || (rc = of_class(Int<2>{})) || (rc = of_class(Int<3>{})) ||
      (rc = of_class(Int<4>{})) || (rc = of_class(Int<5>{})) || (rc = of_class(Int<6>{})) || (rc = of_class(Int<7>{})))
    return rc;
  CB_CUDA(h, cudaFuncSetAttribute(k_phase_a_huge<kOneSeed>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                  static_cast<int>(kSplitSmem)));
  CB_CUDA(h, cudaFuncSetAttribute(k_phase_a_large<kOneSeed>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                  static_cast<int>(kLargeSmem)));
  CB_CUDA(h, cudaFuncSetAttribute(k_phase_a_small<kOneSeed>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                  static_cast<int>(small_smem())));
  CB_CUDA(h, cudaFuncSetAttribute(k_resolve<kMedThreads, kOneSeed>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                  static_cast<int>(resolve_smem<kMedThreads>(kBlockMaxCap, 0))));
  CB_CUDA(h, cudaFuncSetAttribute(k_resolve<kBigThreads, kOneSeed>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                  static_cast<int>(resolve_smem<kBigThreads>(kSmemMaxCap, 2 * int64_t(kSmemMaxCap)))));
  CB_CUDA(h, cudaFuncSetAttribute(k_resolve<kMedThreads, kOneSeed>, cudaFuncAttributePreferredSharedMemoryCarveout,
                                  cudaSharedmemCarveoutMaxShared));
  // shared memory, not L1, limits how many CTAs of these kernels an SM holds
  CB_CUDA(h, cudaFuncSetAttribute(k_phase_a_block<kMedThreads, kOneSeed>,
                                  cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared));
  CB_CUDA(h, cudaFuncSetAttribute(k_phase_a_small<kOneSeed>, cudaFuncAttributePreferredSharedMemoryCarveout,
                                  cudaSharedmemCarveoutMaxShared));
  return CB_OK;
}
}  // namespace

int init_trade_kernels(Graph* h) {
  // the largest dynamic shared memory any handle may ask of each kernel
  int rc = init_seed_kernels<true>(h);
  if (rc || (rc = init_seed_kernels<false>(h))) return rc;
  CB_CUDA(h, cudaFuncSetAttribute(k_retry<kBigThreads>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                  static_cast<int>(resolve_smem<kBigThreads>(kSmemMaxCap, 2 * int64_t(kSmemMaxCap)))));
  CB_CUDA(h, cudaFuncSetAttribute(k_retry_warp, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                  static_cast<int>(WarpWs::kBytes * kWarpWarps)));
  return CB_OK;
}

size_t trade_ws_slice_bytes(int64_t max_trade) {
  return (ws_a_bytes(static_cast<int>(max_trade)) + 255) & ~size_t(255);
}

// Passes of the fix-up: enough that one pass's far-trade records (8 or 16
// bytes per trade) stay below kFixSliceBytes, or the "fix_passes" option.
bool narrow_pack(const Graph* h) { return h->n <= kNarrowPackMax && !h->far_wide; }
constexpr int64_t kFixSliceBytes = int64_t(72) << 20;
int fix_passes(const Graph* h) {
  if (h->fix_passes > 0) return h->fix_passes;
  const int64_t rec = narrow_pack(h) ? 8 : 16;
  return static_cast<int>(std::max<int64_t>(1, (h->ntasks * rec + kFixSliceBytes - 1) / kFixSliceBytes));
}

// Retry passes run where many trades are deferred at once; below kRetryMin
// trades (cb_internal.cuh) the in-order pass alone is faster.
bool small_handle(const Graph* h) { return h->ntasks < kOverlapMax; }
bool runs_retries(const Graph* h) { return h->ntasks >= h->retry_min; }
int retry_passes_of(const Graph* h) { return runs_retries(h) ? h->retry_passes : 0; }

// The next step's permutation and class lists need nothing of this step's
// trades.  With another step to come they are computed beside the in-order
// pass, which leaves most SMs idle (of handles above the one-kernel form, the
// scatter beside the end of the first pass).  Step time n=2^12 71.6 -> 63.3 us,
// 2^14 141 -> 123, 2^15 182 -> 168, 2^16 211 -> 191, 2^17 286 -> 260, 2^18 442 ->
// 423, 2^20 1273 -> 1258; from 2^20 trades on nothing is left of it.
constexpr int64_t kAheadMax = int64_t(1) << 20;
bool may_run_ahead(int64_t ntasks, int64_t nnz) { return nnz > 0 && ntasks < kAheadMax; }
bool runs_ahead(const Graph* h) { return h->order2 && !h->relaxed && !h->timing && !h->swap_stats; }

int super_step(Graph* h, bool ahead) {
  if (h->g >= 0xfffffffeull) return fail(h, CB_ERANGE, "super-step counter exhausted");
  cudaStream_t s = h->stream;
  const int cur = h->cur, nxt = 1 - cur;
  const int eset = h->ev_set;
  cudaEvent_t* ev = h->ev[eset];
  if (h->timing && h->ev_pending[eset]) {
    const int frc = flush_timing(h, eset, true);
    if (frc) return frc;
  }
  StepCtx c;
  c.n = h->n;
  c.T = h->T;
  c.ntasks = h->ntasks;
  c.segs = h->segs;
  c.seg_of = h->seg_of;
  c.rp = h->rp[cur];
  c.col = h->col[cur];
  c.fb = h->stash;
  c.ph = h->col[nxt];
  c.order = h->order[cur];
  c.pos = h->pos[cur];
  c.order_next = h->order[nxt];
  c.pos_next = h->pos[nxt];
  c.rp_next = h->rp[nxt];
  c.chunk_row = h->chunk_row;
  c.thr_key = h->thr_key;
  c.thr_tb = h->thr_tb;
  c.far_pack = h->far_wide ? h->far_wide : h->far_pack;
  c.done = h->done;
  c.err = h->err;
  c.def_bits = h->def_bits;
  c.def_seg = h->def_seg;
  const int64_t nwords = (h->ntasks + 31) / 32;
  const int64_t seg_words = std::max<int64_t>(1, (nwords + kDefSegs - 1) / kDefSegs);
  c.def_seg_trades = 32 * seg_words;
  c.narrow = narrow_pack(h);
  c.seed = h->hsegs[0].seed;   // both used only when the handle holds one graph
  philox_round_keys(c.seed, c.ks);
  // counters (kCtr* in cb_internal.cuh), zero at the start of the step: class
  // lists, deferrals per pass, ranges claimed, global-workspace trades
  int64_t* cnt = h->counters + cur * kCounters;
  unsigned long long* ucnt = reinterpret_cast<unsigned long long*>(cnt);
  c.gws_count = ucnt + kCtrGws;
  const StepEnd end{h->segs, h->nseg, ahead ? nullptr : h->counters + nxt * kCounters,
                    reinterpret_cast<unsigned long long*>(h->counters) + 2 * kCounters, h->def_seg};
  const int64_t ntasks = h->ntasks;
  const int tile_max = h->tile_paths ? std::min(h->tile_max, kTileMaxCap) : 0;
  const int block_max = std::max(h->block_max, tile_max);
  // size classes (L up to 32, 64, tile_max, 256, 512, block_max <= 1024, 2048,
  // min(4096, smem_max), larger); "cta_paths" 0 sends everything above the
  // warp class to the
  // shared-memory kernels (256 threads up to block_max, 1024 above)
  ClassArgs ca;
  ca.n = h->n;
  ca.ntasks = ntasks;
  ca.rp = c.rp;
  ca.lists = h->lists;
  ca.ctr = cnt;
  ClassTh& th = ca.th;
  {
    const int lreg = std::min(TeamCfg<kBigThreads>::kMax, h->smem_max);
    const int t3 = h->cta_paths ? std::max(tile_max, std::min(block_max, TeamCfg<256>::kMax)) : block_max;
    const int t5 = h->cta_paths ? std::max(t3, lreg) : t3;
    th.th[0] = h->lane_teams ? std::min(LaneCfg<8>::Ws::kLmax, tile_max) : 0;
    th.th[1] = h->lane_teams ? std::min(LaneCfg<16>::Ws::kLmax, tile_max) : 0;
    th.th[2] = tile_max;
    th.th[3] = h->cta_paths ? std::min(std::max(TeamCfg<64>::kMax, tile_max), t3) : tile_max;
    th.th[4] = h->cta_paths ? std::min(std::max(TeamCfg<128>::kMax, th.th[3]), t3) : tile_max;
    th.th[5] = t3;
    th.th[6] = h->cta_paths ? std::min(std::max(TeamCfg<512>::kMax, t3), t5) : t3;
    th.th[7] = t5;
  }
  // the next step's permutation and row offsets, and this step's class lists
  if (h->timing) CB_CUDA(h, cudaEventRecord(ev[0], s));
  int rc = CB_OK;
  if (!h->ahead && (rc = compute_permutation(h, 1, -1, h->order[nxt], h->pos[nxt], h->rp[nxt], &ca))) return rc;
  h->ahead = false;
  if (h->timing) CB_CUDA(h, cudaEventRecord(ev[1], s));
  auto launched = [&]() -> int {
    CB_CUDA(h, cudaGetLastError());
    ++h->launches;
    return CB_OK;
  };
  auto finish = [&]() -> int {
    if (ahead) {
      std::swap(h->order[cur], h->order2);
      std::swap(h->pos[cur], h->pos2);
      std::swap(h->rp[cur], h->rp2);
      std::swap(h->chunk_row, h->chunk_row2);
      h->ahead = true;
    }
    h->cur = nxt;
    h->g += 1;
    return CB_OK;
  };
  if (h->nnz == 0) {   // nothing to trade
    k_step_end<<<1, 256, 0, s>>>(end);
    if ((rc = launched())) return rc;
    return finish();
  }
  const int64_t max_trade = 2 * h->maxdeg;
  const size_t med_smem_st = block_smem_bytes(std::max(block_max, 1));   // threshold kernels with staging
  const size_t big_smem_st =
      std::max(block_smem_bytes(std::max(h->smem_max, 1)), max_trade > h->smem_max ? kSplitSmem : 0);
  // the workspace's part of it, before the staging buffer
  auto room_of = [](size_t smem, int stage) { return (smem - (static_cast<size_t>(stage) + 8) * 4) & ~size_t(127); };
  const unsigned mgrid = static_cast<unsigned>(h->num_sms * 4);
  const unsigned bgrid = static_cast<unsigned>(std::max(1, std::min(h->num_sms, h->ws_ctas)));
  const unsigned wgrid = static_cast<unsigned>(h->num_sms * 8);
  // resident CTAs, at most one per trade
  const unsigned small_grid = static_cast<unsigned>(std::min<int64_t>(mgrid, ntasks));
  const unsigned large_grid = static_cast<unsigned>(std::min<int64_t>(h->num_sms, ntasks));
  char* gws = static_cast<char*>(h->ws_global);
  c.cand_max = h->cand_max;
  c.wait_ns = h->wait_ns;
  c.hold_publish = h->hold_publish;
  c.inorder_ctas = h->inorder_ctas ? static_cast<unsigned>(h->inorder_ctas) : ~0u;
  const int32_t* L = h->lists;
  // the first pass: one kernel for classes 0 to 5 and one for 6 and 7, or one
  // per class (large graphs), and the largest trades (no trade is larger than
  // twice the largest degree: classes above that are not launched); a trade
  // whose dependency has not published yet is deferred.  With "timing" on,
  // events ev[4] .. ev[13] bracket the classes' kernels.
  const bool fused = ntasks < h->fuse_max, overlap = small_handle(h);
  auto mark = [&](int k) -> int {
    if (h->timing) CB_CUDA(h, cudaEventRecord(ev[4 + k], s));
    return CB_OK;
  };
  // the kernels come in a one-graph version (the seed's Philox round keys in
  // the kernel parameters) and a general one
  auto run_classes_as = [&](auto one_seed) -> int {
    constexpr bool kOne = decltype(one_seed)::value;
    int r;
    auto run_class = [&](auto k) -> int {
      constexpr int K = decltype(k)::value;
      int rk;
      if ((rk = mark(K))) return rk;
      if ((K > 0 && max_trade <= th.th[K > 0 ? K - 1 : 0]) || (K < 2 && !h->lane_teams)) return CB_OK;
      using Cfg = ClassCfg<K>;
      const unsigned grid = static_cast<unsigned>(h->num_sms * (K < 3 ? 8 : Cfg::kCtas));
      CB_CUDA(h, launch(overlap, k_phase_a_class<K, kOne>, grid, Cfg::kThreads, Cfg::smem(), s, c, L, cnt));
      return launched();
    };
    if (fused) {
      if ((r = mark(0))) return r;
      CB_CUDA(h, launch(overlap, k_phase_a_small<kOne>, small_grid, 256, small_smem(), s, c, L, cnt,
                        (h->lane_teams ? kRunLanes : 0) | (h->cta_paths ? kRunTeams : 0)));
      if ((r = launched())) return r;
      for (int k = 1; k < 6; ++k)
        if ((r = mark(k))) return r;
    } else {
      if ((r = run_class(Int<0>{})) || (r = run_class(Int<1>{})) || (r = run_class(Int<2>{}))) return r;
      if (h->cta_paths && ((r = run_class(Int<3>{})) || (r = run_class(Int<4>{})) || (r = run_class(Int<5>{})))) return r;
      for (int k = 3; k < 6 && !h->cta_paths; ++k)
        if ((r = mark(k))) return r;
    }
    if (!h->cta_paths) {
      k_phase_a_block<kMedThreads, kOne><<<mgrid, kMedThreads, med_smem_st, s>>>(c, L, cnt, 5, block_max,
                                                                         room_of(med_smem_st, block_max), gws,
                                                                                h->ws_slice, block_max);
      if ((r = launched()) || (r = mark(6)) || (r = mark(7))) return r;
    } else if (fused) {
      if ((r = mark(6))) return r;
      if (max_trade > th.th[5]) {
        CB_CUDA(h, launch(overlap, k_phase_a_large<kOne>, large_grid, kBigThreads, kLargeSmem, s, c, L, cnt));
        if ((r = launched())) return r;
      }
      if ((r = mark(7))) return r;
    } else if ((r = run_class(Int<6>{})) || (r = run_class(Int<7>{}))) {
      return r;
    }
    if ((r = mark(8))) return r;
    // the largest trades: in registers up to 8192 entries, the hash in shared
    // memory above; without the register kernels up to smem_max entries in
    // shared memory, staged by a bulk copy
    if (max_trade > th.th[7]) {
      if (h->cta_paths)
        CB_CUDA(h, launch(overlap, k_phase_a_huge<kOne>, bgrid, kBigThreads, kSplitSmem, s, c, L, cnt, h->smem_max, gws,
                          h->ws_slice));
      else
        CB_CUDA(h, launch(overlap, k_phase_a_block<kBigThreads, kOne>, bgrid, kBigThreads, big_smem_st, s, c, L, cnt, 8,
                          h->smem_max, room_of(big_smem_st, h->smem_max), gws, h->ws_slice, h->smem_max));
      if ((r = launched())) return r;
    }
    return mark(9);
  };
  // the first pass over every trade, then the deferred ones: retry passes over
  // their lists, and the in-order pass over what those leave.  Pass r counts
  // its deferrals in ctr[kCtrDef + 3 r ..]
  const int retries = retry_passes_of(h);
  const unsigned lgrid = static_cast<unsigned>(h->num_sms * 4);
  auto defers_to = [&](int r) {
    c.def_n = ucnt + kCtrDef + kDefKinds * r;
    c.def_list = r == retries ? nullptr : (r & 1) ? h->lists : h->def_list;   // the class lists are free after the first pass
  };
  defers_to(0);
  if ((rc = c.seg_of ? run_classes_as(std::false_type{}) : run_classes_as(std::true_type{}))) return rc;
  for (int r = 0; r < retries; ++r) {
    const int32_t* in = c.def_list;
    const unsigned long long* count = c.def_n;
    defers_to(r + 1);
    unsigned long long* claim = ucnt + kCtrClaim + kDefKinds * r;
    k_retry_warp<<<wgrid, 32 * kWarpWarps, WarpWs::kBytes * kWarpWarps, s>>>(c, in, count, claim);
    if ((rc = launched())) return rc;
    if (max_trade > kDefSmall) {
      k_retry<kMedThreads><<<lgrid, kMedThreads, TeamCfg<kMedThreads>::Ws::kBytes, s>>>(c, in + pair_place(1, 0, ntasks), count + 1,
                                                                                       claim + 1, 0, 0, nullptr, 0);
      if ((rc = launched())) return rc;
    }
    if (max_trade > kDefMedium) {
      const size_t sm = resolve_smem<kBigThreads>(h->smem_max, max_trade);
      k_retry<kBigThreads><<<bgrid, kBigThreads, sm, s>>>(c, in + pair_place(2, 0, ntasks), count + 2, claim + 2, h->smem_max, sm, gws,
                                                          h->ws_slice);
      if ((rc = launched())) return rc;
    }
  }
  if (ahead && (rc = compute_permutation(h, 2, -1, h->order2, h->pos2, h->rp2, nullptr, PermPart::kScatterAhead))) return rc;
  if (h->timing) CB_CUDA(h, cudaEventRecord(ev[5 + kClasses], s));
  {
    const bool big = h->inorder_threads == kBigThreads;
    const unsigned grid = big ? bgrid : static_cast<unsigned>(gws ? std::min(h->num_sms * 4, h->ws_ctas) : h->num_sms * 4);
    const int nsegs = static_cast<int>((nwords + seg_words - 1) / seg_words);
    int32_t* list = h->def_list;
    int32_t* chunk_first = h->def_list + ntasks;
    CB_CUDA(h, launch(overlap, k_def_list, nsegs, kDefListThreads, 0, s, c, nwords, nsegs, static_cast<int>(grid), list,
                      chunk_first, ucnt + kCtrChunks, ahead ? h->counters + nxt * kCounters : nullptr));
    if ((rc = launched())) return rc;
    if (big) {
      const size_t sm = resolve_smem<kBigThreads>(h->smem_max, max_trade);
      CB_CUDA(h, launch(overlap, c.seg_of ? k_resolve<kBigThreads, false> : k_resolve<kBigThreads, true>, grid,
                        kBigThreads, sm, s, c, list, chunk_first,
                        ucnt + kCtrChunks, ucnt + kCtrFinished, h->smem_max, sm, gws, h->ws_slice));
    } else {
      const size_t sm = resolve_smem<kMedThreads>(block_max, max_trade);
      CB_CUDA(h, launch(overlap, c.seg_of ? k_resolve<kMedThreads, false> : k_resolve<kMedThreads, true>, grid,
                        kMedThreads, sm, s, c, list, chunk_first,
                        ucnt + kCtrChunks, ucnt + kCtrFinished, block_max, sm, gws, h->ws_slice));
    }
    if ((rc = launched())) return rc;
  }
  if (ahead) {
    ClassArgs next = ca;
    next.rp = h->rp[nxt];
    next.ctr = h->counters + nxt * kCounters;
    if ((rc = compute_permutation(h, 2, -1, h->order2, h->pos2, h->rp2, &next, PermPart::kRestAhead))) return rc;
  }
  if (h->timing) CB_CUDA(h, cudaEventRecord(ev[2], s));
  // rebuild: the fix-up in passes over slices of the far trades; its output
  // overwrites this step's adjacency, which phase A no longer needs, and
  // becomes step g+1's
  {
    const int64_t nnz = h->nnz;
    const int64_t nchunks = (nnz + kFixChunk - 1) / kFixChunk;
    const int passes = fix_passes(h);
    const int64_t per = (ntasks + passes - 1) / passes;
    const unsigned fgrid = static_cast<unsigned>(std::min<int64_t>(nchunks, h->fix_ctas ? h->fix_ctas : h->num_sms * 4));
    int32_t* out = h->col[cur];
    for (int q = 0; q < passes; ++q) {
      const uint32_t lo = static_cast<uint32_t>(std::min<int64_t>(ntasks, q * per));
      const uint32_t hi = static_cast<uint32_t>(std::min<int64_t>(ntasks, (q + 1) * per));
      const bool last = q == passes - 1;
      auto fk = c.narrow ? (last ? k_fixup<true, true> : k_fixup<true, false>)
                         : (last ? k_fixup<false, true> : k_fixup<false, false>);
      CB_CUDA(h, launch(overlap, fk, fgrid, kFixThreads, 0, s, c, nnz, lo, hi, c.ph, c.fb, out, end));
      if ((rc = launched())) return rc;
    }
    std::swap(h->col[0], h->col[1]);   // the step's output is now the other side of the ping-pong
  }
  if (h->timing) {
    CB_CUDA(h, cudaEventRecord(ev[3], s));
    h->ev_pending[eset] = true;
    h->ev_set = 1 - eset;
  }
  return finish();
}

int flush_timing(Graph* h, int set, bool add) {
  if (!h->ev_pending[set]) return CB_OK;
  h->ev_pending[set] = false;
  cudaEvent_t* ev = h->ev[set];
  CB_CUDA(h, cudaEventSynchronize(ev[3]));
  if (!add) return CB_OK;
  float a = 0, b = 0, d = 0, tot = 0;
  CB_CUDA(h, cudaEventElapsedTime(&a, ev[0], ev[1]));
  CB_CUDA(h, cudaEventElapsedTime(&b, ev[1], ev[2]));
  CB_CUDA(h, cudaEventElapsedTime(&d, ev[2], ev[3]));
  CB_CUDA(h, cudaEventElapsedTime(&tot, ev[0], ev[3]));
  h->phase_ms[0] += a;
  h->phase_ms[1] += b;
  h->phase_ms[2] += d;
  h->phase_ms[3] += tot;
  for (int k = 0; k < kClasses; ++k) {
    float e = 0;
    CB_CUDA(h, cudaEventElapsedTime(&e, ev[4 + k], ev[5 + k]));
    h->phase_ms[4 + k] += e;
  }
  float re = 0, io = 0;
  CB_CUDA(h, cudaEventElapsedTime(&re, ev[4 + kClasses], ev[5 + kClasses]));
  CB_CUDA(h, cudaEventElapsedTime(&io, ev[5 + kClasses], ev[2]));
  h->phase_ms[4 + kClasses] += re;
  h->phase_ms[5 + kClasses] += io;
  return CB_OK;
}

}  // namespace cb

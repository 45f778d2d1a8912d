// Edge presence series and their autocorrelation (Section 5.1, "Mixing of
// Edge-Switching, Curveball and Global Curveball").
//
// With the "presence" option a handle keeps, for every node pair {a, b}
// (a < b, local ids) of every graph, one bit per recorded state: bit t of
// the pair's series is set when the edge exists after the t-th recorded super
// step (t = 0: the state when recording started).  cb_autocorr classifies each
// pair that ever occurred: for thinning k, the transitions of the k-thinned
// series (entries 0, k, 2k, ...) are fitted to an independent and to a
// first-order Markov model, and the edge counts as correlated when the
// Markov model fits better by the Bayesian information criterion,
// G^2 = 2 (L_Markov - L_independent) > ln N over its N transitions (the
// criterion is the reading of this library; the paper cites it without
// printing it).  A constant series, and one with fewer than two thinned
// transitions, counts as independent.
#include <algorithm>
#include <cmath>
#include <vector>

#include "cb_internal.cuh"

namespace cb {

struct PresenceBufs {
  int64_t T = 0;             // super steps the record holds after its step 0
  int64_t t = 0;             // states recorded so far
  int64_t W = 0;             // 32-bit words per pair
  int64_t pairs = 0;         // pairs over every graph
  uint32_t* bits = nullptr;  // pairs x W
  int64_t* base = nullptr;   // device: first pair of each graph
  size_t bytes = 0;          // device bytes of bits and base
  std::vector<int64_t> hbase;
};

namespace {

__device__ __forceinline__ int64_t pair_index(int64_t n, int64_t a, int64_t b) {
  return a * n - a * (a + 1) / 2 + (b - a - 1);
}

// One warp per position: every entry (x, y) with x < y (local ids) sets
// bit t of its pair.
__global__ void k_presence(int64_t npos, const int32_t* __restrict__ order, const int64_t* __restrict__ rp,
                           const int32_t* __restrict__ col, const Seg* __restrict__ segs,
                           const int32_t* __restrict__ seg_of, const int64_t* __restrict__ base, int64_t W,
                           int64_t t, uint32_t* __restrict__ bits) {
  const int lane = threadIdx.x & 31;
  const int64_t warps = static_cast<int64_t>(gridDim.x) * (blockDim.x >> 5);
  for (int64_t p = (blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x) >> 5; p < npos; p += warps) {
    const int g = seg_of ? seg_of[p] : 0;
    const int64_t off = segs[g].off, n = segs[g].n;
    const int64_t x = order[p] - off;
    for (int64_t e = rp[p] + lane; e < rp[p + 1]; e += 32) {
      const int64_t y = order[col[e]] - off;
      if (x < y && y < n) {
        const int64_t q = base[g] + pair_index(n, x, y);
        atomicOr(bits + q * W + (t >> 5), 1u << (t & 31));
      }
    }
  }
}

__device__ __forceinline__ double xlogy(double a, double b) { return a == 0.0 ? 0.0 : a * log(a / b); }

// One warp per pair of graph g: lane l classifies thinnings k = l + 1 and
// k = l + 33.  out[0..kmax) correlated pairs, out[64..64+kmax) decisions
// within 1e-9 of the boundary, out[128] pairs that occurred.
__global__ void k_autocorr(int64_t npairs, int64_t first, int64_t W, int64_t states, int kmax,
                           const uint32_t* __restrict__ bits, unsigned long long* __restrict__ out) {
  __shared__ unsigned long long acc[129];
  for (int i = threadIdx.x; i < 129; i += blockDim.x) acc[i] = 0;
  __syncthreads();
  const int lane = threadIdx.x & 31;
  const int64_t warps = static_cast<int64_t>(gridDim.x) * (blockDim.x >> 5);
  for (int64_t q = (blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x) >> 5; q < npairs; q += warps) {
    const uint32_t* s = bits + (first + q) * W;
    bool any = false;
    for (int64_t i = lane; i < W; i += 32) any |= __ldg(s + i) != 0u;
    if (!__any_sync(0xffffffffu, any)) continue;
    if (lane == 0) atomicAdd(&acc[128], 1ull);
    for (int r = 0; r < 2; ++r) {
      const int k = lane + 1 + 32 * r;
      if (k > kmax) continue;
      // thinned entries x_0 .. x_N at steps 0, k, ..., N k
      const int64_t N = (states - 1) / k;
      if (N < 2) continue;
      int64_t ones_head = 0, ones_tail = 0, n11 = 0;   // ones among x_0..x_{N-1}, among x_1..x_N, pairs (1,1)
      int prev = static_cast<int>(__ldg(s) & 1u);
      for (int64_t j = 1; j <= N; ++j) {
        const int64_t st = j * k;
        const int cur = static_cast<int>((__ldg(s + (st >> 5)) >> (st & 31)) & 1u);
        ones_head += prev;
        ones_tail += cur;
        n11 += prev & cur;
        prev = cur;
      }
      const double n10 = static_cast<double>(ones_head - n11), n01 = static_cast<double>(ones_tail - n11);
      const double d11 = static_cast<double>(n11), dN = static_cast<double>(N);
      const double n00 = dN - d11 - n10 - n01;
      const double r0 = n00 + n01, r1 = n10 + n11;           // rows: x_{s-1} = 0, 1
      const double c0 = n00 + n10, c1 = n01 + n11;           // columns: x_s = 0, 1
      const double l1 = xlogy(n00, r0) + xlogy(n01, r0) + xlogy(n10, r1) + xlogy(d11, r1);
      const double l0 = xlogy(c0, dN) + xlogy(c1, dN);
      const double m = 2.0 * (l1 - l0) - log(dN);
      if (m > 0.0) atomicAdd(&acc[k - 1], 1ull);
      if (fabs(m) < 1e-9) atomicAdd(&acc[64 + k - 1], 1ull);
    }
  }
  __syncthreads();
  for (int i = threadIdx.x; i < 129; i += blockDim.x)
    if (acc[i]) atomicAdd(&out[i], acc[i]);
}

// The same classification for records of at most kFixedStates states, bound
// by integer instructions instead of FP64 logarithms (seven per pair and
// thinning, on a chip with almost no FP64) and a loop over the transitions:
//   - the transition counts are population counts of the series' words: with
//     the mask of the thinned positions, ones among x_0..x_{N-1} and pairs
//     (1,1) as series & (series >> k);
//   - every term of G^2 is i ln i for a count i <= N, read from a table in
//     fixed point (rounded from long double), so G^2 is a sum of integers.
//     The scale keeps the largest value below 2^61.  Nine terms, rounded by up
//     to half a unit and doubled, and ln N leave G^2 - ln N within 9.5 units of
//     its exact value: 5.4e-13 at 8192 states, 8.4e-15 at 301.  The largest
//     errors over 200000 random tables are 4.3e-13 and 6.3e-15; the FP64
//     formula's on the same tables are 5.3e-12 and 2.2e-13.
// 8 graphs of 2000 nodes, 301 states, kmax 32: the whole pass (300 super
// steps, record, classification) went from 212 to 69 ms, all but 5 ms of it
// here.
constexpr int kFixedStates = 8192;
constexpr int kFixedThreads = 512;

// Fraction bits of the fixed point for counts below `states`.
int fixed_shift(int64_t states) {
  const double top = states > 2 ? static_cast<double>(states) * std::log(static_cast<double>(states)) : 2.0;
  return 60 - std::ilogb(top);
}

size_t fixed_smem(int64_t states, int64_t W, int kmax) {
  return sizeof(int64_t) * static_cast<size_t>(states + kmax) + sizeof(uint32_t) * static_cast<size_t>(W * kmax);
}

__global__ void __launch_bounds__(kFixedThreads) k_autocorr_fixed(int64_t npairs, int64_t first, int W, int states,
                                                                 int kmax, int64_t near,
                                                                 const int64_t* __restrict__ xlnx,
                                                                 const uint32_t* __restrict__ bits,
                                                                 unsigned long long* __restrict__ out) {
  extern __shared__ uint64_t tab[];              // i ln i, i < states; then ln N of each k; then the masks
  uint64_t* lnn = tab + states;
  uint32_t* head = reinterpret_cast<uint32_t*>(lnn + kmax);   // word w of thinning k: head[w kmax + k - 1]
  __shared__ unsigned int acc[129];
  for (int i = threadIdx.x; i < 129; i += blockDim.x) acc[i] = 0;
  for (int i = threadIdx.x; i < states + kmax; i += blockDim.x) tab[i] = static_cast<uint64_t>(xlnx[i]);
  for (int i = threadIdx.x; i < W * kmax; i += blockDim.x) {
    const int w = i / kmax, k = i % kmax + 1;
    const int end = (states - 1) / k * k;        // the last thinned position (not of the head)
    uint32_t m = 0;
    for (int p = (32 * w + k - 1) / k * k; p < 32 * w + 32 && p < end; p += k) m |= 1u << (p - 32 * w);
    head[i] = m;
  }
  __syncthreads();
  const int lane = threadIdx.x & 31;
  const int64_t warps = static_cast<int64_t>(gridDim.x) * (blockDim.x >> 5);
  for (int64_t q = (blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x) >> 5; q < npairs; q += warps) {
    const uint32_t* s = bits + (first + q) * W;
    bool any = false;
    for (int i = lane; i < W; i += 32) any |= __ldg(s + i) != 0u;
    if (!__any_sync(0xffffffffu, any)) continue;
    if (lane == 0) atomicAdd(&acc[128], 1u);
    for (int k = lane + 1; k <= kmax; k += 32) {
      const int N = (states - 1) / k;
      if (N < 2) continue;
      const int wofs = k >> 5, sh = k & 31;
      int ones = 0, n11 = 0;
      uint32_t lo = wofs < W ? __ldg(s + wofs) : 0u;
      for (int w = 0; w < W; ++w) {
        const uint32_t x = __ldg(s + w) & head[w * kmax + k - 1];
        const uint32_t hi = w + wofs + 1 < W ? __ldg(s + w + wofs + 1) : 0u;
        ones += __popc(x);
        n11 += __popc(x & __funnelshift_r(lo, hi, sh));   // bits p + k of the series
        lo = hi;
      }
      const int last = N * k;
      const int tail = ones - static_cast<int>(__ldg(s) & 1u) + static_cast<int>((__ldg(s + (last >> 5)) >> (last & 31)) & 1u);
      const int n10 = ones - n11, n01 = tail - n11, n00 = N - n11 - n10 - n01;
      // partial sums may wrap; G^2 / 2 itself is at most N ln 2
      const uint64_t g = tab[n00] + tab[n01] + tab[n10] + tab[n11] + tab[N] - tab[N - ones] - tab[ones] -
                         tab[N - tail] - tab[tail];
      const int64_t m = static_cast<int64_t>(2 * g - lnn[k - 1]);
      if (m > 0) atomicAdd(&acc[k - 1], 1u);
      if (m <= near && m >= -near) atomicAdd(&acc[64 + k - 1], 1u);   // |G^2 - ln N| < 1e-9
    }
  }
  __syncthreads();
  for (int i = threadIdx.x; i < 129; i += blockDim.x)
    if (acc[i]) atomicAdd(&out[i], static_cast<unsigned long long>(acc[i]));
}

// i ln i for i < states in fixed point, then ln N for N = (states - 1) / k, k = 1..kmax.
std::vector<int64_t> fixed_table(int64_t states, int kmax) {
  const long double one = std::ldexp(1.0L, fixed_shift(states));
  std::vector<int64_t> t;
  t.reserve(static_cast<size_t>(states + kmax));
  for (int64_t i = 0; i < states; ++i)
    t.push_back(i == 0 ? 0 : std::llroundl(static_cast<long double>(i) * std::log(static_cast<long double>(i)) * one));
  for (int k = 1; k <= kmax; ++k)
    t.push_back(std::llroundl(std::log(static_cast<long double>(std::max<int64_t>((states - 1) / k, 1))) * one));
  return t;
}

}  // namespace

void free_presence(Graph* h) {
  if (!h->pres) return;
  if (h->pres->bits) cudaFreeAsync(h->pres->bits, h->stream);
  if (h->pres->base) cudaFreeAsync(h->pres->base, h->stream);
  h->dev_bytes -= static_cast<int64_t>(h->pres->bytes);
  delete h->pres;
  h->pres = nullptr;
}

int record_presence(Graph* h) {
  PresenceBufs* b = h->pres;
  if (!b || b->t > b->T) return CB_OK;   // off, or full
  if (h->n > 0) {
    const unsigned grid = static_cast<unsigned>(std::min<int64_t>((h->n + 7) / 8, int64_t(h->num_sms) * 16));
    k_presence<<<grid, 256, 0, h->stream>>>(h->n, h->order[h->cur], h->rp[h->cur], h->col[h->cur], h->segs,
                                           h->seg_of, b->base, b->W, b->t, b->bits);
    CB_CUDA(h, cudaGetLastError());
    ++h->launches;
  }
  b->t += 1;
  return CB_OK;
}

int set_presence(Graph* h, int64_t T) {
  free_presence(h);
  if (T == 0) return CB_OK;
  PresenceBufs* b = new (std::nothrow) PresenceBufs;
  if (!b) return fail(h, CB_ENOMEM, "host allocation failed");
  b->T = T;
  b->W = (T + 1 + 31) / 32;
  b->hbase.resize(h->nseg);
  int64_t pairs = 0;
  for (int g = 0; g < h->nseg; ++g) {
    b->hbase[g] = pairs;
    const int64_t n = h->hsegs[g].n;
    pairs += n * (n - 1) / 2;
  }
  b->pairs = pairs;
  const double bytes = static_cast<double>(pairs) * static_cast<double>(b->W) * 4.0;
  if (bytes > 64e9) {
    delete b;
    return fail(h, CB_EINVAL, "presence record above 64 GB (pairs x steps too large)");
  }
  const size_t nbits = std::max<size_t>(static_cast<size_t>(bytes), 4), nbase = sizeof(int64_t) * h->nseg;
  void* p = nullptr;
  void* q = nullptr;
  if (dev_alloc(h, &p, nbits)) {
    delete b;
    return fail(h, CB_ENOMEM, "device allocation failed (presence record)");
  }
  if (dev_alloc(h, &q, nbase)) {
    cudaFreeAsync(p, h->stream);
    h->dev_bytes -= static_cast<int64_t>(nbits);
    delete b;
    return fail(h, CB_ENOMEM, "device allocation failed (presence record)");
  }
  b->bits = static_cast<uint32_t*>(p);
  b->base = static_cast<int64_t*>(q);
  b->bytes = nbits + nbase;
  h->pres = b;
  CB_CUDA(h, cudaMemsetAsync(b->bits, 0, static_cast<size_t>(bytes), h->stream));
  CB_CUDA(h, cudaMemcpyAsync(b->base, b->hbase.data(), sizeof(int64_t) * h->nseg, cudaMemcpyHostToDevice,
                             h->stream));
  CB_CUDA(h, cudaStreamSynchronize(h->stream));   // hbase is read by the copy
  return record_presence(h);                       // step 0: the current state
}

}  // namespace cb

extern "C" int cb_autocorr(cb_handle h, int32_t graph, int32_t kmax, int64_t* correlated, int64_t* near_ties,
                           int64_t* occurring, int64_t* states) {
  using namespace cb;
  if (!h || kmax < 1 || kmax > 64 || !correlated) return fail(h, CB_EINVAL, "bad argument (kmax in [1, 64])");
  if (!h->pres) return fail(h, CB_EINVAL, "no presence record (set the \"presence\" option first)");
  if (graph < -1 || graph >= h->nseg) return fail(h, CB_EINVAL, "graph index out of range");
  if (h->latched) return fail(h, h->latched, "handle has a latched error: " + h->last_error);
  PresenceBufs* b = h->pres;
  const int64_t used = std::min(b->t, b->T + 1);
  unsigned long long* d = nullptr;
  if (dev_alloc(h, reinterpret_cast<void**>(&d), 129 * sizeof(unsigned long long)))
    return fail(h, CB_ENOMEM, "device allocation failed");
  CB_CUDA(h, cudaMemsetAsync(d, 0, 129 * sizeof(unsigned long long), h->stream));
  const int g0 = graph < 0 ? 0 : graph, g1 = graph < 0 ? h->nseg : graph + 1;
  std::vector<int64_t> table;
  int64_t* dtable = nullptr;
  const bool fixed = used <= kFixedStates && b->W <= kFixedStates / 32;
  if (fixed) {
    table = fixed_table(used, kmax);
    if (dev_alloc(h, reinterpret_cast<void**>(&dtable), table.size() * sizeof(int64_t))) {
      cudaFreeAsync(d, h->stream);
      h->dev_bytes -= 129 * sizeof(unsigned long long);
      return fail(h, CB_ENOMEM, "device allocation failed");
    }
    CB_CUDA(h, cudaMemcpyAsync(dtable, table.data(), table.size() * sizeof(int64_t), cudaMemcpyHostToDevice,
                               h->stream));
    CB_CUDA(h, cudaFuncSetAttribute(k_autocorr_fixed, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                    static_cast<int>(fixed_smem(kFixedStates, kFixedStates / 32, 64))));
  }
  for (int g = g0; g < g1; ++g) {
    const int64_t n = h->hsegs[g].n, np = n * (n - 1) / 2;
    if (np == 0) continue;
    if (fixed) {
      const size_t sm = fixed_smem(used, b->W, kmax);
      const unsigned grid = static_cast<unsigned>(std::min<int64_t>((np + 15) / 16, int64_t(h->num_sms) * 8));
      k_autocorr_fixed<<<grid, kFixedThreads, sm, h->stream>>>(np, b->hbase[g], static_cast<int>(b->W),
                                                              static_cast<int>(used), kmax,
                                                              static_cast<int64_t>(std::ldexp(1e-9, fixed_shift(used))),
                                                              dtable, b->bits, d);
      CB_CUDA(h, cudaGetLastError());
      ++h->launches;
      continue;
    }
    const unsigned grid = static_cast<unsigned>(std::min<int64_t>((np + 7) / 8, int64_t(h->num_sms) * 16));
    k_autocorr<<<grid, 256, 0, h->stream>>>(np, b->hbase[g], b->W, used, kmax, b->bits, d);
    CB_CUDA(h, cudaGetLastError());
    ++h->launches;
  }
  unsigned long long hv[129];
  CB_CUDA(h, cudaMemcpyAsync(hv, d, sizeof(hv), cudaMemcpyDeviceToHost, h->stream));
  CB_CUDA(h, cudaStreamSynchronize(h->stream));
  cudaFreeAsync(d, h->stream);
  h->dev_bytes -= 129 * sizeof(unsigned long long);
  if (dtable) {
    cudaFreeAsync(dtable, h->stream);
    h->dev_bytes -= static_cast<int64_t>(table.size() * sizeof(int64_t));
  }
  for (int k = 0; k < kmax; ++k) {
    correlated[k] = static_cast<int64_t>(hv[k]);
    if (near_ties) near_ties[k] = static_cast<int64_t>(hv[64 + k]);
  }
  if (occurring) *occurring = static_cast<int64_t>(hv[128]);
  if (states) *states = used;
  return check_device_error(h);
}

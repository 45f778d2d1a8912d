// Trade size classes: every trade falls into one of kClasses classes (by
// L = deg u + deg v against ascending thresholds), each run by its own team
// size.  The lists are built by the permutation kernels of the same super
// step: they read the current step's row offsets and the permutation the next
// step's keys, so neither waits for the other and no launch is spent on them.
#pragma once
#include "cb_internal.cuh"
#include "pair_lists.cuh"
#include "team.cuh"

namespace cb {

struct ClassTh {
  int th[kClasses - 1];   // class k holds th[k-1] < L <= th[k] (th[-1] = -1, th[kClasses-1] = inf)
};

struct ClassArgs {
  int64_t n, ntasks;     // ntasks 0: nothing to classify
  const int64_t* rp;     // row offsets of the current step
  ClassTh th;
  int32_t* lists;        // two classes to an array of ntasks (pair_lists.cuh)
  int64_t* ctr;          // zeroed counters: kCtrClsLen, kCtrFirstEnt
};

// Chunks of trades a CTA classifies at a time: one trade per thread while
// that leaves work for every CTA, eight (an eighth of the atomics on the list
// lengths) for large graphs.
inline int class_per(int64_t ntasks) { return ntasks > (int64_t(1) << 18) ? 8 : 1; }
inline int64_t class_chunks(int64_t ntasks, int threads) {
  const int64_t c = int64_t(threads) * class_per(ntasks);
  return (ntasks + c - 1) / c;
}

// Chunks first, first + stride, ... by a CTA of NT threads: per
// class one reservation of list space per chunk; a chunk's trades stay
// together, roughly in index order, so their rows are neighbours in memory.
template <int NT, int PER>
__device__ void classify_chunks(const ClassArgs& a, int64_t first, int64_t stride) {
  __shared__ int cnt[kClasses];
  __shared__ int put[kClasses];
  __shared__ unsigned long long ent[kClasses];
  __shared__ int64_t base[kClasses];
  const int lane = threadIdx.x & 31;
  const unsigned below = (1u << lane) - 1u;
  constexpr int64_t kChunk = int64_t(NT) * PER;
  for (int64_t ch = first; ch * kChunk < a.ntasks; ch += stride) {
    if (threadIdx.x < kClasses) {
      cnt[threadIdx.x] = put[threadIdx.x] = 0;
      ent[threadIdx.x] = 0;
    }
    __syncthreads();
    int8_t cls[PER];
#pragma unroll
    for (int j = 0; j < PER; ++j) {
      const int64_t t = ch * kChunk + j * NT + threadIdx.x;
      int k = -1, L = 0;
      if (t < a.ntasks) {
        const int64_t b0 = a.rp[2 * t], b1 = a.rp[2 * t + 1];
        const int64_t b2 = 2 * t + 1 < a.n ? a.rp[2 * t + 2] : b1;
        L = static_cast<int>(b2 - b0);
        k = 0;
#pragma unroll
        for (int i = 0; i < kClasses - 1; ++i) k += L > a.th.th[i];
      }
      cls[j] = static_cast<int8_t>(k);
#pragma unroll
      for (int q = 0; q < kClasses; ++q) {
        const unsigned b = __ballot_sync(kFull, k == q);
        if (!b) continue;
        const unsigned e = __reduce_add_sync(kFull, k == q ? static_cast<unsigned>(L) : 0u);
        if (lane == 0) {
          atomicAdd(&cnt[q], __popc(b));
          atomicAdd(&ent[q], static_cast<unsigned long long>(e));
        }
      }
    }
    __syncthreads();
    if (threadIdx.x < kClasses && cnt[threadIdx.x]) {
      unsigned long long* c = reinterpret_cast<unsigned long long*>(a.ctr);
      base[threadIdx.x] = static_cast<int64_t>(
          atomicAdd(c + kCtrClsLen + threadIdx.x, static_cast<unsigned long long>(cnt[threadIdx.x])));
      atomicAdd(c + kCtrFirstEnt + threadIdx.x, ent[threadIdx.x]);
    }
    __syncthreads();
#pragma unroll
    for (int j = 0; j < PER; ++j) {
      const int64_t t = ch * kChunk + j * NT + threadIdx.x;
      const int k = cls[j];
#pragma unroll
      for (int q = 0; q < kClasses; ++q) {
        const unsigned b = __ballot_sync(kFull, k == q);
        if (!b) continue;
        int p = 0;
        if (lane == 0) p = atomicAdd(&put[q], __popc(b));
        p = __shfl_sync(kFull, p, 0);
        if (k == q) a.lists[pair_place(q, base[q] + p + __popc(b & below), a.ntasks)] = static_cast<int32_t>(t);
      }
    }
    __syncthreads();
  }
}

template <int NT>
__device__ __forceinline__ void classify(const ClassArgs& a, int64_t first, int64_t stride) {
  if (a.ntasks > (int64_t(1) << 18)) classify_chunks<NT, 8>(a, first, stride);
  else classify_chunks<NT, 1>(a, first, stride);
}

}  // namespace cb

// The two run queues of the uniform-trade executor in one array of as many
// places as there are trades: small trades from the front, large ones from the
// back (pair_lists.cuh).  Plain C++ apart from the qualifiers, so that it also compiles for the
// host.
#pragma once
#include <cstdint>

#include "pair_lists.cuh"

namespace cb {

struct RunQueues {
  int64_t trades, large;   // places; how many of them are for large trades
  __host__ __device__ int64_t length(int big) const { return big ? large : trades - large; }
  // Is place q in this queue?  (Past its length it would be the other's.)
  __host__ __device__ bool holds(int big, uint64_t q) const { return q < static_cast<uint64_t>(length(big)); }
  __host__ __device__ int64_t place(int big, uint64_t q) const { return pair_place(big, static_cast<int64_t>(q), trades); }
};

}  // namespace cb

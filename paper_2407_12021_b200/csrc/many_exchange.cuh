// Which of its two exchange buffers a couple of warps of the GEMM for calls of many rows uses (gemm_many.cu; plain C++, so that a test on
// the host can include it).
#pragma once

namespace aded {

// Per exchange the two warps write, meet at a barrier and read what the other wrote.  One that is through may write the next exchange
// while its partner still reads this one, so two exchanges in a row must not use the same buffer -- also the last of one item and the
// first of the next, between which nothing else holds the warps together.  Hence a count over all of a warp's exchanges, not
// one per item: an item has an odd number of them with blocks of 160 and 224 rows.
struct ManyExchange {
    int count = 0;
#ifdef __CUDACC__
    __device__ __forceinline__
#endif
    int next() { return count++ & 1; }
};

}  // namespace aded

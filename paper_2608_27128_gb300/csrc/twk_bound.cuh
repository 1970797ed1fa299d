// twk_bound.cuh -- the word by which one thread of the audit's epilogue tells another the best
// value it has found for their row (twk_audit.cu): a lower bound on the row's maximum in the
// segment at hand, and that segment's stamp, in 32 bits.
//
// The value gives its low 5 bits to the stamp modulo 32, so what is read back is the value
// rounded down (it is positive): still a lower bound, and what stays below it cannot be the
// row's maximum.  The reader takes it only under the stamp of its own segment.  A thread
// clears its word when it enters a segment, two segments make a work item, and the two result
// buffers let neither thread be three items ahead of the other: what the reader can see of the
// word is at most seven stamps from its own, and 32 are told apart.
#pragma once
#include <cstdint>

namespace twk {

constexpr uint32_t kBoundStamp = 31u;         // the bits that carry the stamp
constexpr uint32_t kNoBound = 0xFF800000u;    // the bits of -inf

// The word for the positive float whose bits are v (or for -inf: no bound).
__host__ __device__ constexpr uint32_t bound_word(uint32_t v, uint32_t stamp)
{
    return (v & ~kBoundStamp) | (stamp & kBoundStamp);
}

// The bits of the float that `word` gives as a bound in segment `stamp`.
__host__ __device__ constexpr uint32_t bound_bits(uint32_t word, uint32_t stamp)
{
    return ((word ^ stamp) & kBoundStamp) == 0u ? word & ~kBoundStamp : kNoBound;
}

}  // namespace twk

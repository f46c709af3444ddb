// Sums of the vectors of a limb GEMM whose matrix holds its digits centred.
#pragma once
#include <cstdint>

namespace qpadl {

// Digits are stored centred, as d - p / 2 for d in [0, p), p at most 256: of magnitude 128 at most, and small ones keep
// the tensor cores' power down (digits of 0 and 1 stored as -128 and -127 cost 21696 x 23488 with 174 queries 4%).
constexpr uint32_t digit_centre(uint32_t p) { return p / 2; }
// Columns per partial sum of a vector.
constexpr uint32_t kSumCols = 2048;
__host__ __device__ constexpr uint32_t limb_sum_parts(uint64_t cols) {
    return static_cast<uint32_t>((cols + kSumCols - 1) / kSumCols);
}
// The sum mod 2^32 of vector v is that of words[x * nv + v] over x < parts.
struct VecSums {
    const uint32_t *words;
    uint32_t nv, parts, centre;
#ifdef __CUDACC__
    // What centring took from every output of vector v.  The kernels load it as a tile starts, beside its MMAs,
    // one vector per lane: loaded at a tile's end it cost 2 us a tile (6000 x 600, 320 vectors, two tiles one
    // after the other, 23.1 us; 19.3 this way).  Not a read-only load: the words come from the kernel that a
    // programmatic dependent overlaps.
    __device__ __forceinline__ uint32_t centred(uint32_t v) const {
        uint32_t s = 0;
#pragma unroll 8
        for (uint32_t x = 0; x < parts; ++x) s += __ldcg(words + (uint64_t)x * nv + v);
        return centre * s;
    }
#endif
};

}  // namespace qpadl

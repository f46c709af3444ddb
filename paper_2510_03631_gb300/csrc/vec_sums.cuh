// Sums of the vectors of a limb GEMM whose matrix holds its digits centred.
#pragma once
#include <cstdint>

namespace qpadl {

// Digits are stored centred, as d - 128.
constexpr uint32_t kCentre = 128;
// Columns per partial sum of a vector.
constexpr uint32_t kSumCols = 2048;
__host__ __device__ constexpr uint32_t limb_sum_parts(uint64_t cols) {
    return static_cast<uint32_t>((cols + kSumCols - 1) / kSumCols);
}
// The sum mod 2^32 of vector v is that of words[x * nv + v] over x < parts.
struct VecSums {
    const uint32_t *words;
    uint32_t nv, parts;
#ifdef __CUDACC__
    // What centring took from every output of vector v.  The kernels load it as a tile starts, beside its MMAs,
    // one vector per lane: loaded at a tile's end it cost 2 us a tile (6000 x 600, 320 vectors, two tiles one
    // after the other, 23.1 us; 19.3 this way).  Not a read-only load: the words come from the kernel that a
    // programmatic dependent overlaps.
    __device__ __forceinline__ uint32_t centred(uint32_t v) const {
        uint32_t s = 0;
#pragma unroll 8
        for (uint32_t x = 0; x < parts; ++x) s += __ldcg(words + (uint64_t)x * nv + v);
        return kCentre * s;
    }
#endif
};

}  // namespace qpadl

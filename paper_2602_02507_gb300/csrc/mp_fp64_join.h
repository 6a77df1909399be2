// mp_fp64_join.h -- the integer sum of one chain's accumulators (mp_fp64_tc.cu), plain C++.
//
// Accumulator s of a chain of up to 128 terms is an integer x_s with |x_s| <= (s + 1) 2^21, of weight
// 2^(8 (5 - s)) in units of the sixth; the sixth arrives with the seventh, divided by 2^DS, as x_5.
// The sum is formed modulo 2^64 from 32-bit words that carry offsets, so that pairs of them
// are put together in 32 unsigned bits:
//   a_0, a_1, a_2, a_5: x + kFloatOff, the bits of 1.5 2^23 + x, for |x| <= 2^22
//   a_3: x + 2^23;  a_4: x
// Each pair stays within [0, 2^32) modulo the offsets' own overflow:
//   a_2 256 + a_3 = 2^30 + 256 x_2 + x_3 + 2^23       in [0, 2^31 + 2^24]
//   a_4 (256 / 2^DS) + a_5 = kFloatOff + ...          in [kFloatOff - 2^29.4, kFloatOff + 2^29.4], DS >= 2
//   a_0 256 + a_1 = 2^30 + 256 x_0 + kFloatOff + x_1  in [2^30, 2^32)
#pragma once
#include <cstdint>

#ifdef __CUDACC__
#define MP_HD __host__ __device__ __forceinline__
#else
#define MP_HD inline
#endif

namespace mp {

constexpr uint32_t kFloatOff = 0x4B400000u;     // bits of 1.5 2^23
constexpr uint32_t kThirdPairOff = 0x00800000u;  // 2^23, on a_3

template <int DS>
struct ChainJoin {
    // what the offsets add to the sum, modulo 2^64
    static constexpr uint32_t p01 = kFloatOff * 257u, p23 = kFloatOff * 256u + kThirdPairOff;  // modulo 2^32
    static constexpr uint64_t offset =
        (uint64_t)p23 * (65536u >> DS) + kFloatOff + (uint64_t)p01 * ((1ull << 32) >> DS);
    static MP_HD uint64_t sum(uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t a4, uint32_t a5)
    {
        return (uint64_t)(a2 * 256u + a3) * (65536u >> DS) + (a4 * (256u >> DS) + a5) +
               (uint64_t)(a0 * 256u + a1) * ((1ull << 32) >> DS);
    }
};

}  // namespace mp

// Sum of the 32 floats of a warp without the FP64 pipe (1/64 of the FP32
// rate), with at least the accuracy of FP64 additions.
//
// A float is an integer of 24 bits times a power of two.  Shifted to the
// largest exponent of the warp with 34 bits below it, the 32 integers add
// exactly in 64 bits; only what lies more than 2^57 below the largest value is
// cut off (FP64 additions round at 2^-53 of every partial sum).  The sum of
// three limbs of 27, 27 and 10 bits is three 32-bit warp reductions.
//
// In k_chan_adj, whose two sums per warp these are, the slots they are added
// to loaded ahead: 41.3 ms per gradient of 500 steps of 128x64x64 nodes, 4.52
// of 160 steps of 48x20x24; two-float sums by shuffles (about 46 bits) with the
// slots loaded at the end 42.2 and 4.54.
#pragma once

#include <stdint.h>

#ifdef __CUDACC__
#define LBM_HD __host__ __device__ __forceinline__
#else
#define LBM_HD inline
#endif

namespace lbm {

constexpr int kSumBits = 34;

// Exponent field of a float's bits, that of the smallest normal number for
// zeros and subnormal ones.
LBM_HD int sum_exp(uint32_t u) {
    const int e = (int)((u >> 23) & 255u);
    return e ? e : 1;
}

// The float as a multiple of 2^(E - 150 - kSumBits), E >= its exponent.
LBM_HD long long sum_fixed(uint32_t u, int E) {
    const long long m = (long long)((u & 0x7fffffu) | ((u >> 23) & 255u ? 0x800000u : 0u)) << kSumBits;
    const int sh = E - sum_exp(u);
    const long long a = sh < 64 ? m >> sh : 0;
    return (int32_t)u < 0 ? -a : a;
}

// A 64-bit integer as limbs that 32 of them add up in 32 bits: two of 27 bits
// without a sign, the rest with it.
LBM_HD uint32_t sum_lo(long long a) { return (uint32_t)a & 0x7ffffffu; }
LBM_HD uint32_t sum_mid(long long a) { return (uint32_t)(a >> 27) & 0x7ffffffu; }
LBM_HD int32_t sum_hi(long long a) { return (int32_t)(a >> 54); }

// The total of the limbs.
LBM_HD long long sum_total(uint32_t lo, uint32_t mid, int32_t hi) {
    return (long long)((unsigned long long)(long long)hi << 54) + ((long long)mid << 27) + (long long)lo;
}

// The bits of 2^(E - 150 - kSumBits).
LBM_HD long long sum_unit_bits(int E) { return (long long)(E - 150 - kSumBits + 1023) << 52; }

#ifdef __CUDACC__
// Sums of a and b over the warp; lane 0 returns that of a, lane 1 that of b
// (the other lanes either).  Infinities and NaN take the FP64 additions.
__device__ __forceinline__ double warp_sum2(const float a, const float b) {
    const uint32_t ua = __float_as_uint(a), ub = __float_as_uint(b), all = 0xffffffffu;
    const int Ea = __reduce_max_sync(all, sum_exp(ua)), Eb = __reduce_max_sync(all, sum_exp(ub));
    const bool second = threadIdx.x & 1;
    if (Ea == 255 || Eb == 255) {
        double x = a, y = b;
        for (int o = 16; o > 0; o >>= 1) {
            x += __shfl_xor_sync(all, x, o);
            y += __shfl_xor_sync(all, y, o);
        }
        return second ? y : x;
    }
    const long long fa = sum_fixed(ua, Ea), fb = sum_fixed(ub, Eb);
    const uint32_t la = __reduce_add_sync(all, sum_lo(fa)), lb = __reduce_add_sync(all, sum_lo(fb));
    const uint32_t ma = __reduce_add_sync(all, sum_mid(fa)), mb = __reduce_add_sync(all, sum_mid(fb));
    const int32_t ha = __reduce_add_sync(all, sum_hi(fa)), hb = __reduce_add_sync(all, sum_hi(fb));
    const long long t = second ? sum_total(lb, mb, hb) : sum_total(la, ma, ha);
    return (double)t * __longlong_as_double(sum_unit_bits(second ? Eb : Ea));
}
#endif

}  // namespace lbm

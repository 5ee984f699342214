// Philox-2x64 with 10 rounds (Salmon, Moraes, Dror, Shaw, "Parallel random
// numbers: as easy as 1, 2, 3", SC'11), the counter-based generator the paper
// takes from Random123 for its random fields (Sec. 2).  Per round the first
// counter word is multiplied by the published 64-bit multiplier; the new first
// word is hi(product) xor key xor second word, the new second word
// lo(product); the key advances by the published Weyl increment.
//
// The 64 x 64 -> 128-bit product is a 128-bit integer product on both sides: on
// the device that measured 5.45 ps a draw over a full GPU against 5.66 for
// __umul64hi with a 64-bit multiply and 6.0-7.3 for sums of four 32 x 32 ->
// 64-bit products (the wide multiplications bound it: 40 a draw).  The header
// compiles for the host too, where a test checks it against the generator's
// published known answers.
#pragma once

#include <stdint.h>

#if defined(__CUDACC__)
#define TL_PHILOX_FN __host__ __device__ __forceinline__
#else
#define TL_PHILOX_FN inline
#endif

namespace tl {

// (hi, lo) = a * b for a, b < 2^64.
TL_PHILOX_FN void mul_64x64_128(uint64_t a, uint64_t b, uint64_t &hi, uint64_t &lo)
{
    const unsigned __int128 p = (unsigned __int128)a * b;
    hi = (uint64_t)(p >> 64);
    lo = (uint64_t)p;
}

// Rounds r0 .. 9 on (c0, c1).
template <int R0>
TL_PHILOX_FN void philox2x64_rounds(uint64_t c0, uint64_t c1, uint64_t key, uint64_t &o0, uint64_t &o1)
{
    const uint64_t M = 0xD2B74407B1CE6E93ULL;
    const uint64_t Wk = 0x9E3779B97F4A7C15ULL;
    key += R0 * Wk;
#pragma unroll
    for (int r = R0; r < 10; ++r) {
        uint64_t hi, lo;
        mul_64x64_128(M, c0, hi, lo);
        c0 = hi ^ key ^ c1;
        c1 = lo;
        key += Wk;
    }
    o0 = c0;
    o1 = c1;
}

TL_PHILOX_FN void philox2x64_10(uint64_t c0, uint64_t c1, uint64_t key, uint64_t &o0, uint64_t &o1)
{
    philox2x64_rounds<0>(c0, c1, key, o0, o1);
}

// The same for a first counter word below 2^32: its first product takes two of
// the four wide multiplications.
TL_PHILOX_FN void philox2x64_10_low(uint32_t c0, uint64_t c1, uint64_t key, uint64_t &o0, uint64_t &o1)
{
    const uint64_t low = (uint64_t)0xB1CE6E93u * c0, high = (uint64_t)0xD2B74407u * c0 + (low >> 32);
    philox2x64_rounds<1>((high >> 32) ^ key ^ c1, (high << 32) | (uint32_t)low, key, o0, o1);
}

}  // namespace tl

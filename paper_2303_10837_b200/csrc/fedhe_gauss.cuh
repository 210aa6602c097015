// Discrete Gaussian samples from 64-bit uniform words through a small table.
#pragma once

#include "fedhe_device.cuh"

namespace fedhe {

// ---------------------------------------------------------------------------
// discrete Gaussian, sigma = 3.2 on [-19, 19]: thresholds floor(2^64 Pr[X <= x])
// for x = -19 .. 18; a 64-bit uniform r maps to -19 + #{x : r >= T[x]}
// ---------------------------------------------------------------------------
#define FEDHE_GAUSS_CDF { \
    0x0000000bd798c7acull, 0x00000053f5e234f7ull, 0x000001e24b89625aull, 0x000009adbc7900e1ull, \
    0x00002d17ca1e3a82ull, 0x0000bf05ff772ee2ull, 0x0002e06843bbf95dull, 0x000a19062dceb033ull, \
    0x00204c0ded173b17ull, 0x005e3163ffc656a8ull, 0x00fab6a7e614dfaeull, 0x0261b16e99bc14f8ull, \
    0x054c69348bbc9867ull, 0x0acd276539458231ull, 0x143796b3c337f00bull, 0x22d43df09de40e7aull, \
    0x37651d96aa4fb429ull, 0x51a5da2b40f1bff1ull, 0x700ad4bf5a6e80e2ull, 0x8ff52b40a5917f1dull, \
    0xae5a25d4bf0e400eull, 0xc89ae26955b04bd6ull, 0xdd2bc20f621bf185ull, 0xebc8694c3cc80ff4ull, \
    0xf532d89ac6ba7dceull, 0xfab396cb74436798ull, 0xfd9e4e916643eb07ull, 0xff05495819eb2051ull, \
    0xffa1ce9c0039a957ull, 0xffdfb3f212e8c4e8ull, 0xfff5e6f9d2314fccull, 0xfffd1f97bc4406a2ull, \
    0xffff40fa0088d11dull, 0xffffd2e835e1c57dull, 0xfffff6524386ff1eull, 0xfffffe1db4769da5ull, \
    0xffffffac0a1dcb08ull, 0xfffffff428673853ull}
#if defined(__CUDACC__)
static __constant__ uint64_t c_gauss_cdf[38] = FEDHE_GAUSS_CDF;
#endif
HD uint64_t gauss_threshold(int x) {
#if !defined(__CUDA_ARCH__)
    constexpr uint64_t c_gauss_cdf[38] = FEDHE_GAUSS_CDF;
#endif
    return c_gauss_cdf[x];
}

HD int gauss_from_u64(uint64_t r) {
    int v = -19;
#if defined(__CUDA_ARCH__)
#pragma unroll
#endif
    for (int x = 0; x < 38; x++) v += (r >= gauss_threshold(x)) ? 1 : 0;
    return v;
}

// The same map through shared-memory tables, by the high word of r alone.  An entry belongs to one value of r's top
// byte, or of its second byte where the top one is 00 or ff (these hold most of the thresholds): in the top byte of
// the entry the number of thresholds certainly not above r, below it 2^24 less the next 24 bits of the one threshold that shares
// the entry's range.  Adding the next 24 bits of r carries into the top byte when r is not below that threshold, so a
// sample costs one 4-byte load, an addition and a shift.  Not decided are ranges with more than one threshold
// (1 sample in 32,768) and sums whose low 24 bits are close to a carry, where bits that are not in the word count: behind
// the second byte it has 16 bits and not 24, so up to 255 may be missing (1 in 65,536).  With the bytes 00
// and ff undecided (1 sample in 128) two calls of five had a lane that needed the whole block.
struct alignas(16) GaussTables {
    uint32_t entry[3 * 256];         // by the top byte; by the second byte behind 00; by the second byte behind ff
};
constexpr uint32_t GAUSS_UNDECIDED = 0x80000000u;

HD uint32_t gauss_entry(uint64_t lo, int width) {        // r in [lo, lo + 2^width)
    const uint64_t last = lo + ((1ull << width) - 1);
    uint32_t base = 0, in = 0;
    uint64_t t_in = 0;
#if defined(__CUDA_ARCH__)
#pragma unroll 1
#endif
    for (int x = 0; x < 38; x++) {
        const uint64_t t = gauss_threshold(x);
        if (t <= lo) base++;
        else if (t <= last) { in++; t_in = t; }
    }
    if (in > 1) return GAUSS_UNDECIDED;
    return (base << 24) + (in ? (1u << 24) - ((uint32_t)(t_in >> (width - 24)) & 0xffffffu) : 0u);
}

HD void gauss_tables_init(GaussTables &g, uint32_t tid, uint32_t nthreads) {
    for (uint32_t i = tid; i < 768; i += nthreads) {
        const uint32_t row = i >> 8;
        const uint64_t b = i & 255u;
        g.entry[i] = row == 0 ? gauss_entry(b << 56, 56) : gauss_entry((row == 2 ? 0xffull << 56 : 0) | (b << 48), 48);
    }
}

// value + 19 in the top byte, unless gauss_undecided(); hi: the high word of r
HD uint32_t gauss_sum(const GaussTables &g, uint32_t hi) {
    const bool edge = hi + 0x01000000u < 0x02000000u;                  // top byte ff or 00
    const uint32_t at = edge ? 256u + ((hi >> 16) & 511u) : hi >> 24;  // bit 24 tells ff from 00
    return g.entry[at] + ((edge ? hi << 8 : hi) & 0xffffffu);
}
HD bool gauss_undecided(uint32_t sum) { return (int)sum < 0 || ((sum + 255u) & 0xffffffu) < 256u; }

}  // namespace fedhe

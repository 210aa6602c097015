// Shared by the kernel files of the library: launch bookkeeping, the error
// samplers, small modular helpers, the per-limb choice of arithmetic and the
// outer stages of the long transforms.
#pragma once

#include "fedhe_gauss.cuh"
#include "fedhe_launch.h"

#include <atomic>
#include <type_traits>

namespace fedhe {

extern std::atomic<uint64_t> g_launches;      // kernels launched by this library (fedhe_transform.cu)

#define FEDHE_LAUNCHED() (g_launches.fetch_add(1), cudaGetLastError())

static inline unsigned blocks_for(size_t count, unsigned per_block) {
    return (unsigned)((count + per_block - 1) / per_block);
}

// Words 1 and 3 of a stream block, the high halves of its two 64-bit values.  The last round makes them from two
// low products, and the round before it only has to make the factors of these.
__device__ __forceinline__ uint2 stream_block_high(uint64_t seed, uint32_t block, uint32_t t, uint32_t client, uint32_t tag_limb) {
    uint32_t k0 = (uint32_t)seed, k1 = (uint32_t)(seed >> 32);
    u32x4 c = {block, t, client, tag_limb};
#pragma unroll
    for (int r = 0; r < 9; r++) {
        uint32_t h0, l0, h1, l1;
        mulhilo32(0xD2511F53u, c.x, h0, l0);
        mulhilo32(0xCD9E8D57u, c.z, h1, l1);
        c = u32x4{h1 ^ c.y ^ k0, l1, h0 ^ c.w ^ k1, l0};
        k0 += 0x9E3779B9u;
        k1 += 0xBB67AE85u;
    }
    return make_uint2(0xCD9E8D57u * c.z, 0xD2511F53u * c.x);
}

// a copy of the context's table (768 entries from 38 thresholds each took 3 us of every call)
__device__ __forceinline__ void gauss_tables_load(GaussTables &g, const void *made, uint32_t tid, uint32_t nthreads) {
    for (uint32_t i = tid; i < sizeof(GaussTables) / 16; i += nthreads)
        reinterpret_cast<uint4 *>(&g)[i] = __ldg(static_cast<const uint4 *>(made) + i);
}

static __device__ __noinline__ int2 gauss_pair_whole(uint64_t seed, uint32_t block, uint32_t t, uint32_t client, uint32_t tag) {
    const u32x4 w = stream_block(seed, block, t, client, tag);
    const uint64_t a = (uint64_t)w.x | ((uint64_t)w.y << 32), b = (uint64_t)w.z | ((uint64_t)w.w << 32);
    int2 v = make_int2(-19, -19);
#pragma unroll 1
    for (int x = 0; x < 38; x++) {
        v.x += (a >= c_gauss_cdf[x]) ? 1 : 0;
        v.y += (b >= c_gauss_cdf[x]) ? 1 : 0;
    }
    return v;
}
// The two samples of each of the stream blocks block + j * step, j < U, side by side: a block by itself is a chain of
// ten products.  Only the high words decide nearly always, so the generator's last two rounds make no others (stream_block_high).
template <int U>
__device__ __forceinline__ void gauss_pairs(int2 (&v)[U], const GaussTables &g, uint64_t seed, uint32_t block, uint32_t step,
                                            uint32_t t, uint32_t client, uint32_t tag) {
    uint2 hi[U];
#pragma unroll
    for (int j = 0; j < U; j++) hi[j] = stream_block_high(seed, block + j * step, t, client, tag);
#pragma unroll
    for (int j = 0; j < U; j++) {
        const uint32_t s0 = gauss_sum(g, hi[j].x), s1 = gauss_sum(g, hi[j].y);
        v[j] = make_int2((int)(s0 >> 24) - 19, (int)(s1 >> 24) - 19);
        if (gauss_undecided(s0) || gauss_undecided(s1)) v[j] = gauss_pair_whole(seed, block + j * step, t, client, tag);
    }
}
__device__ __forceinline__ int2 gauss_pair(const GaussTables &g, uint64_t seed, uint32_t block, uint32_t t, uint32_t client,
                                           uint32_t tag) {
    int2 v[1];
    gauss_pairs<1>(v, g, seed, block, 0, t, client, tag);
    return v[0];
}

__device__ __forceinline__ uint64_t addmod(uint64_t a, uint64_t b, uint64_t q) { return csub(a + b, q); }
__device__ __forceinline__ uint64_t submod(uint64_t a, uint64_t b, uint64_t q) { return a >= b ? a - b : a + q - b; }

// slow exact helpers, used only when keys and key shares are made
static __device__ uint64_t mod_u128(uint64_t hi, uint64_t lo, uint64_t q) {
    uint64_t r = 0;
    for (int i = 63; i >= 0; i--) { r = (r << 1) | ((hi >> i) & 1); r = csub(r, q); }
    for (int i = 63; i >= 0; i--) { r = (r << 1) | ((lo >> i) & 1); r = csub(r, q); }
    return r;
}
static __device__ uint64_t mulmod_slow(uint64_t a, uint64_t b, uint64_t q) {
    return mod_u128(__umul64hi(a, b), a * b, q);
}
static __device__ uint64_t shoup_companion(uint64_t w, uint64_t q) {   // floor(w 2^64 / q), w < q
    uint64_t rem = w, quo = 0;
    for (int i = 0; i < 64; i++) {
        rem <<= 1; quo <<= 1;
        if (rem >= q) { rem -= q; quo |= 1; }
    }
    return quo;
}

// A limb runs in double-precision arithmetic when its prime allows it.
#define FEDHE_FOR_ARITH(lb, CALL)                               \
    if ((lb).fwd_d) { using M_ = ModF64; CALL; }                \
    else { using M_ = ModInt; CALL; }

// the same with the select flavour of the integer arithmetic (kernels bound by the multiply pipe)
#define FEDHE_FOR_ARITH_SEL(lb, CALL)                           \
    if ((lb).fwd_d) { using M_ = ModF64; CALL; }                \
    else { using M_ = ModIntSel; CALL; }

// The A = logN - LOGB outer stages of a long transform on two neighbouring
// columns of the 2^A x B matrix view (x[a], y[a] = row a): forward from
// canonical input, inverse with 1/N folded into stage 0.
template <uint32_t A, class M>
__device__ __forceinline__ void outer_forward(typename M::val (&x)[1u << A], typename M::val (&y)[1u << A],
                                              const NttArgsT<M> &t) {
    constexpr uint32_t rows = 1u << A;
#pragma unroll
    for (uint32_t s = 0; s < A; s++) {
        const uint32_t bit = 1u << (A - 1 - s);
#pragma unroll
        for (uint32_t a = 0; a < rows; a++) {
            if (a & bit) continue;
            const auto w = M::load(t.tw + (1u << s) + (a >> (A - s)));
            t.m.fwd(x[a], x[a | bit], w);
            t.m.fwd(y[a], y[a | bit], w);
        }
    }
}

template <uint32_t A, class M, class T>
__device__ __forceinline__ void outer_inverse(typename M::val (&x)[1u << A], typename M::val (&y)[1u << A],
                                              const NttArgsT<M> &t, const T &ninv, const T &wn) {
    constexpr uint32_t rows = 1u << A;
#pragma unroll
    for (int s = (int)A - 1; s >= 1; s--) {
        const uint32_t bit = 1u << (A - 1 - s);
#pragma unroll
        for (uint32_t a = 0; a < rows; a++) {
            if (a & bit) continue;
            const auto w = M::load(t.tw + (1u << s) + (a >> (A - s)));
            t.m.inv(x[a], x[a | bit], w);
            t.m.inv(y[a], y[a | bit], w);
        }
    }
    constexpr uint32_t bit = 1u << (A - 1);      // stage 0 with 1/N folded in
#pragma unroll
    for (uint32_t a = 0; a < rows; a++) {
        if (a & bit) continue;
        t.m.inv_scaled(x[a], x[a | bit], ninv, wn);
        t.m.inv_scaled(y[a], y[a | bit], ninv, wn);
    }
}

// The outer stages as an elementwise pass over HBM: every thread owns two
// neighbouring columns and reads and writes whole 16-byte words.
// launches kern<A> for the context's A (1, 2 or 3)
#define FEDHE_FOR_A(c, CALL)                 \
    switch ((c).A) {                         \
    case 1: { constexpr uint32_t A_ = 1; CALL; } break; \
    case 2: { constexpr uint32_t A_ = 2; CALL; } break; \
    default: { constexpr uint32_t A_ = 3; CALL; } break; \
    }

// the block (inner) stages of a batch of transforms only (fedhe_transform.cu)
cudaError_t launch_ntt_inner(const CtxDev &c, bool forward, uint64_t *data, size_t npoly, size_t poly_stride,
                             uint32_t limb0, uint32_t nlimbs, cudaStream_t s);

}  // namespace fedhe

// Encryption and decryption by complex transforms of split integers (part 7 of the kernels):
// the coefficient format on every ring.  fedhe_fft.cuh has the method and its error bounds.
#include "fedhe_kernels.cuh"
#include "fedhe_slots.cuh"

namespace fedhe {

constexpr double FFT_ROUND = 6755399441055744.0;                 // 1.5 * 2^52: adding it rounds to an integer ...
constexpr int64_t FFT_ROUND_BITS = 0x4338000000000000;           // ... that is the difference of the bit patterns

// integer |v| < 2^51 as a double
__device__ __forceinline__ double fft_from_int(int64_t v) {
    return f64_sub(__longlong_as_double(v + FFT_ROUND_BITS), FFT_ROUND);
}
__device__ __forceinline__ int64_t fft_round_bits(double z) { return __double_as_longlong(f64_add(z, FFT_ROUND)); }

// The thread's number, read anew: what is computed from it cannot be kept in registers across a
// transform, whose sixteen points need them (the kernels would spill addresses instead).
__device__ __forceinline__ uint32_t fresh_tid() {
    uint32_t t;
    asm volatile("mov.u32 %0, %%tid.x;" : "=r"(t));
    return t;
}
// a table entry that passes by: L1 belongs to what is used again
__device__ __forceinline__ double2 load_passing(const double2 *p) {
    double2 v;
    asm("ld.global.nc.L1::no_allocate.v2.f64 {%0, %1}, [%2];" : "=d"(v.x), "=d"(v.y) : "l"(p));
    return v;
}

// Adds to `v` the top piece z of a product (not rounded), weighed 2^shift, less q times the quotient: all
// modulo 2^64, and the top piece has magnitude at most q / 2 and a little then.
struct FftJoin {
    uint64_t minus_q, fix;
    double scale;
    uint32_t shift;
    __device__ __forceinline__ FftJoin(const FftSplit &f, uint64_t q) : FftJoin(q, f.top_scale, f.shift[f.pieces - 1]) {}
    __device__ __forceinline__ FftJoin(uint64_t q, double top_scale, uint32_t top_shift) : minus_q(0 - q), scale(top_scale), shift(top_shift) {
        // the quotient carries 2^17, which keeps it positive
        fix = (q << 17) - ((uint64_t)FFT_ROUND_BITS << shift);
    }
    __device__ __forceinline__ int64_t operator()(int64_t v, double z) const {
        const uint32_t k = (uint32_t)__double_as_longlong(f64_fma(z, scale, FFT_ROUND + 131072.0));
        return (int64_t)((uint64_t)v + fix + ((uint64_t)fft_round_bits(z) << shift) + (uint64_t)k * minus_q);
    }
};

// the residue in [0, q) of |v| < q
__device__ __forceinline__ uint64_t fft_canonical(int64_t v, uint64_t q) {
    if (v < 0) v += (int64_t)q;
    return (uint64_t)v;
}

// geometry of a ring: a cluster of R thread blocks, one per block of the transform
template <int CL_>
struct FftRing {
    using Tab = FftTab<CL_>;
    static constexpr int CL = CL_, R = 1 << CL, NB = FftLay::NB, NT = FftLay::NT, n = R * NB, N = 2 * n;
    static constexpr int PER = 16 / R;     // columns of the R x NB view that a thread finishes
    static constexpr size_t SMEM = (size_t)NB * 16 + (size_t)Tab::WORDS * 16;
};

// a word of the buffer of block `a` of the cluster
template <int CL>
__device__ __forceinline__ cpx buffer_of(const double2 *buf, uint32_t a, uint32_t word) {
    if constexpr (CL == 0) {
        const double2 v = buf[word];
        return cpx{v.x, v.y};
    } else {
        uint32_t at = (uint32_t)__cvta_generic_to_shared(buf + word), there;
        cpx v;
        asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(there) : "r"(at), "r"(a));
        asm volatile("ld.shared::cluster.v2.f64 {%0, %1}, [%2];" : "=d"(v.re), "=d"(v.im) : "r"(there));
        return v;
    }
}

// x = this block's row in layout C -> x[i R + a] = coefficient a NB + tid + NT (rank PER + i): every
// block takes its columns from the buffers of all and runs the stages between blocks on them
template <class G>
__device__ __forceinline__ void fft_gather(cpx (&x)[16], double2 *buf, const root_t *tab, uint32_t rank, uint32_t tid) {
    if constexpr (G::CL > 0) {
#pragma unroll
        for (int r = 0; r < 16; r++) buf[r * G::NT + tid] = make_double2(x[r].re, x[r].im);     // the thread's own words
        cluster_arrive();
        cluster_wait();
#pragma unroll
        for (int i = 0; i < 16; i++)
            x[i] = buffer_of<G::CL>(buf, i % G::R, (rank * G::PER + i / G::R) * G::NT + tid);
    }
    buffer_free<G::CL>();
#pragma unroll
    for (int i = 0; i < G::PER; i++) {
        cpx v[G::R];
#pragma unroll
        for (int a = 0; a < G::R; a++) v[a] = x[i * G::R + a];
        fft_outer_inverse<G::CL>(v, tab, tid, rank * G::PER + i);
#pragma unroll
        for (int a = 0; a < G::R; a++) x[i * G::R + a] = v[a];
    }
}
// The reverse: coefficients of the columns of this block -> this block's row, layout C
template <class G>
__device__ __forceinline__ void fft_spread(cpx (&x)[16], double2 *buf, const root_t *fwd, uint32_t rank, uint32_t tid) {
    if constexpr (G::CL > 0) {
        buffer_wait<G::CL>();
#pragma unroll
        for (int i = 0; i < G::PER; i++) {
            cpx v[G::R];
#pragma unroll
            for (int a = 0; a < G::R; a++) v[a] = x[i * G::R + a];
            fft_outer_forward<G::CL>(v, fwd);
#pragma unroll
            for (int b = 0; b < G::R; b++) buf[(b * G::PER + i) * G::NT + tid] = make_double2(v[b].re, v[b].im);
        }
        cluster_arrive();
        cluster_wait();
#pragma unroll
        for (int r = 0; r < 16; r++)
            x[r] = buffer_of<G::CL>(buf, r / G::PER, (rank * G::PER + r % G::PER) * G::NT + tid);
        buffer_free<G::CL>();
    }
}
// coefficient of value i (0 .. 31: column, row, real or imaginary part) of a thread, less the thread's number
template <class G>
__device__ __forceinline__ uint32_t fft_coefficient(int i, uint32_t rank) {
    const int o = i >> 1;
    return (o % G::R) * G::NB + G::NT * (rank * G::PER + o / G::R) + (i & 1) * G::n;
}
// the value that position i of block `blk` (of 2^LEV) has after LEV stages of the encoder's network
template <int LEV>
__device__ __forceinline__ cpx encoder_stages(const float *slots, const double2 *ftw, uint32_t n, uint32_t blk, uint32_t i) {
    if constexpr (LEV == 0) {
        return cpx{(double)__ldg(slots + i), 0.0};
    } else {
        const uint32_t half = n >> LEV;
        const cpx U = encoder_stages<LEV - 1>(slots, ftw, n, blk >> 1, i);
        const cpx V = encoder_stages<LEV - 1>(slots, ftw, n, blk >> 1, i + half);
        if ((blk & 1u) == 0) return cadd_rn(U, V);
        cpx w = load_ftw(ftw, half + i);
        w.im = -w.im;
        return cmul_rn(csub_rn(U, V), w);
    }
}

// ===========================================================================
// encryption:  c0 = pk0 u + e0 + m,  c1 = pk1 u + e1   (mod every q_j), coefficient format
// ===========================================================================

// ---- tensor memory as a store of the threads' own words ----
//
// The kernel has no matrix products, so its 256 KB of tensor memory per SM would lie idle: each of the two
// thread blocks takes half of it (256 columns), which is 128 words for every thread.  Words kept there
// cost neither L2 nor shared-memory bandwidth.
constexpr uint32_t TMEM_COLS = 256, TMEM_WORDS = 128;

__device__ __forceinline__ uint32_t tmem_take(uint32_t *where) {       // by the whole block
    if (threadIdx.x < 32) {
        const uint32_t at = (uint32_t)__cvta_generic_to_shared(where);
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(at), "n"(TMEM_COLS) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    __syncthreads();
    // a warp reaches the 32 lanes of its number modulo 4; the warps 0..3 and 4..7 share them by columns
    const uint32_t warp = threadIdx.x >> 5;
    return *where + ((warp & 3u) << 21) + (warp >> 2) * TMEM_WORDS;
}
__device__ __forceinline__ void tmem_give(uint32_t base) {             // by the whole block, after its last use
    __syncthreads();
    if (threadIdx.x < 32)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(base), "n"(TMEM_COLS));
}
__device__ __forceinline__ void tmem_put8(uint32_t at, const uint32_t (&w)[8]) {
    asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"r"(at), "r"(w[0]), "r"(w[1]),
                 "r"(w[2]), "r"(w[3]), "r"(w[4]), "r"(w[5]), "r"(w[6]), "r"(w[7])
                 : "memory");
}
__device__ __forceinline__ void tmem_wait_put() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }
__device__ __forceinline__ void tmem_get32(uint32_t at, uint32_t (&w)[32]) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];\n\ttcgen05.wait::ld.sync.aligned;"
                 : "=r"(w[0]), "=r"(w[1]), "=r"(w[2]), "=r"(w[3]),
                 "=r"(w[4]), "=r"(w[5]), "=r"(w[6]), "=r"(w[7]),
                 "=r"(w[8]), "=r"(w[9]), "=r"(w[10]), "=r"(w[11]),
                 "=r"(w[12]), "=r"(w[13]), "=r"(w[14]), "=r"(w[15]),
                 "=r"(w[16]), "=r"(w[17]), "=r"(w[18]), "=r"(w[19]),
                 "=r"(w[20]), "=r"(w[21]), "=r"(w[22]), "=r"(w[23]),
                 "=r"(w[24]), "=r"(w[25]), "=r"(w[26]), "=r"(w[27]),
                 "=r"(w[28]), "=r"(w[29]), "=r"(w[30]), "=r"(w[31])
                 : "r"(at)
                 : "memory");
}
__device__ __forceinline__ cpx tmem_cpx(const uint32_t *w) {
    return cpx{__hiloint2double((int)w[1], (int)w[0]), __hiloint2double((int)w[3], (int)w[2])};
}
__device__ __forceinline__ void tmem_get8(uint32_t at, uint32_t (&w)[8]) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];\n\ttcgen05.wait::ld.sync.aligned;"
                 : "=r"(w[0]), "=r"(w[1]), "=r"(w[2]), "=r"(w[3]), "=r"(w[4]), "=r"(w[5]), "=r"(w[6]), "=r"(w[7])
                 : "r"(at)
                 : "memory");
}
// ---- the key's table comes in through the transform buffer, ahead of its use ----
constexpr uint32_t KEY_BYTES = FftLay::NB * 16;

__device__ __forceinline__ void key_fetch(double2 *buf, const double2 *key, uint64_t *bar) {       // by one thread
    const uint32_t at = (uint32_t)__cvta_generic_to_shared(buf), b = (uint32_t)__cvta_generic_to_shared(bar);
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(b), "n"(KEY_BYTES) : "memory");
    asm volatile("cp.async.bulk.shared::cta.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(at), "l"(key),
                 "n"(KEY_BYTES), "r"(b)
                 : "memory");
}
// whether the copy is there, after 10 ms at most
__device__ __forceinline__ bool key_try(uint64_t *bar, uint32_t parity) {
    const uint32_t b = (uint32_t)__cvta_generic_to_shared(bar);
    uint32_t done;
    asm volatile("{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, 0x989680;\n\tselp.u32 %0, 1, 0, p;\n\t}"
                 : "=r"(done)
                 : "r"(b), "r"(parity)
                 : "memory");
    return done != 0;
}
constexpr uint32_t KEY_TRIES = 256;

// two complex values
__device__ __forceinline__ void tmem_put(uint32_t at, cpx a, cpx b) {
    const uint32_t w[8] = {(uint32_t)__double2loint(a.re), (uint32_t)__double2hiint(a.re), (uint32_t)__double2loint(a.im),
                           (uint32_t)__double2hiint(a.im), (uint32_t)__double2loint(b.re), (uint32_t)__double2hiint(b.re),
                           (uint32_t)__double2loint(b.im), (uint32_t)__double2hiint(b.im)};
    tmem_put8(at, w);
}
__device__ __forceinline__ void tmem_get(uint32_t at, cpx &a, cpx &b) {
    uint32_t w[8];
    tmem_get8(at, w);
    a = cpx{__hiloint2double((int)w[1], (int)w[0]), __hiloint2double((int)w[3], (int)w[2])};
    b = cpx{__hiloint2double((int)w[5], (int)w[4]), __hiloint2double((int)w[7], (int)w[6])};
}

// Scratch in global memory (it lives in L2) and tensor memory of an encryption.
template <int CL_>
struct EncRing {
    using Tab = FftTab<CL_>;
    static constexpr int CL = CL_, R = 1 << CL, NB = FftLay::NB, NT = FftLay::NT, n = R * NB, N = 2 * n;
    static constexpr bool E_IN_SMEM = CL < 2;             // e1 (a byte each) fits beside the buffers of two blocks
    // of the R blocks of a product the last stays in registers or shared memory; so many wait in tensor memory ...
    static constexpr int WAIT_TMEM = R == 1 ? 0 : R == 2 ? 1 : 2, WAIT_L2 = R - 1 - WAIT_TMEM;
    // ... and for R <= 2 the 32-bit products of low pieces do, in the words from PARK_AT; for R = 1 the transform of u, from 0
    static constexpr bool PARK_TMEM = R <= 2;
    static constexpr uint32_t PARK_AT = 64;
    // for R <= 2 those are all there are: of a prime below 2^61 the low piece has 21 bits at most, and 22 fit (cut_limbs() checks)
    static constexpr bool ALL_NARROW = R <= 2;
    static constexpr int COLUMNS = R == 1 ? 4 : R == 2 ? 2 : 1, K = COLUMNS * R * 2;      // columns, values finished together
    // whether what a column needs from L2 is fetched a column ahead: of R = 8 it does not fit the registers
    static constexpr bool FAR_AHEAD = R == 4;
    // a cluster's: the transform of u, the message and e0, flags
    static constexpr size_t UHAT = (size_t)n * 16, TERMS = (size_t)N * 8, SHARED = UHAT + TERMS + 128;
    // a ciphertext's samples: e0, e1 (a byte each), u in two bits each, the rows of a column side by side
    using Row = typename std::conditional<(R <= 4), uint8_t, uint16_t>::type;
    static constexpr size_t E0 = 0, E1 = N, U = 2 * (size_t)N, SAMPLES = U + 2 * NB * sizeof(Row);
    // items of u (four neighbouring columns of a half to a thread, all their rows: 512, 512, 1024, 2048 stream blocks), of either error (512)
    static constexpr uint32_t U_COLUMNS = R == 1 ? 2 : 1, U_ITEMS = 2 * NB / 4 / (NT * U_COLUMNS), E_ITEMS = N / 2 / (2 * NT),
                              ITEMS = U_ITEMS + 2 * E_ITEMS;
    // a thread block's: what waits, joined low pieces
    static constexpr size_t WAIT = (size_t)WAIT_L2 * NB * 16, PARK = ALL_NARROW ? 0 : (size_t)N * 8, OWN = WAIT + PARK;
    static constexpr size_t SMEM = (size_t)NB * 16 + (size_t)Tab::WORDS * 16 + (E_IN_SMEM ? N : 0);
};

// What a thread block needs to know of the products, in shared memory: looked up in the kernel's parameters, by the unit's number, then
// its limb's, it was a chain of misses of 900 clocks before every block of a transform (N = 16384).  Put together from the parameters at the
// start of the kernel it was these misses again, for every product one behind the other (one ciphertext of N = 8192, 8 limbs of
// 60 bits: 24.7 us, 22.3 before that and 22.6 now; 888 of 8 limbs of 45 bits: 645, 650 to 700, 628); one load brings the finished table.
__device__ __forceinline__ void enc_jobs_load(EncJobs &s, const EncJobs *made) {
    static_assert(sizeof(EncJobs) / 16 <= FftLay::NT, "a load for every thread");
    if (threadIdx.x < sizeof(EncJobs) / 16) reinterpret_cast<uint4 *>(&s)[threadIdx.x] = __ldg(reinterpret_cast<const uint4 *>(made) + threadIdx.x);
}

// What a ciphertext's draws depend on besides its number, and whether the clusters draw for themselves.
struct EncDraw { uint64_t seed; uint32_t client, t0, inside; };

// value i (column, row, real or imaginary part) of a thread's columns from r0: its coefficient less the thread's number
template <class G>
__device__ __forceinline__ uint32_t enc_coefficient(uint32_t r0, int i) {
    const int o = i >> 1;
    return (o % G::R) * G::NB + G::NT * (r0 + o / G::R) + (i & 1) * G::n;
}

// What columns need from L2 is fetched ahead: a loop that loads it where it is used waits for every column.
template <class G>
struct EncAhead {
    static constexpr int W = G::WAIT_L2 ? G::WAIT_L2 : 1;
    cpx w[W];                              // the column in the blocks that wait in L2
    int low[G::PARK_TMEM ? 1 : G::K];      // its parked words
    __device__ __forceinline__ void fetch_wait(const double2 *wait, uint32_t r, uint32_t tid) {
#pragma unroll
        for (int a = 0; a < G::WAIT_L2; a++) {
            const double2 v = __ldcg(wait + a * G::NB + r * G::NT + tid);
            w[a] = cpx{v.x, v.y};
        }
    }
    __device__ __forceinline__ void fetch_low(const unsigned char *park, uint32_t r, uint32_t tid) {
        if constexpr (!G::PARK_TMEM) {
            static_assert(G::COLUMNS == 1 && G::K % 4 == 0, "whole 16-byte words of one column");
#pragma unroll
            for (int i = 0; i < G::K; i += 4) {
                const int4 v = __ldcg(reinterpret_cast<const int4 *>(park) + (r * (G::K / 4) + i / 4) * G::NT + tid);
                low[i] = v.x;
                low[i + 1] = v.y;
                low[i + 2] = v.z;
                low[i + 3] = v.w;
            }
        }
    }
};

// Columns r0 .. r0 + COLUMNS - 1 of a product as they enter the stages between blocks ...
template <class G>
__device__ __forceinline__ void enc_columns(cpx (&v)[G::COLUMNS][G::R], const cpx (&x)[16], const double2 *buf, const EncAhead<G> &ahead,
                                            uint32_t tm, uint32_t r0, uint32_t tid) {
    if constexpr (G::R == 1) {
#pragma unroll
        for (int i = 0; i < G::COLUMNS; i++) v[i][0] = x[r0 + i];
    } else if constexpr (G::R == 2) {
        tmem_get(tm + r0 * 4, v[0][0], v[1][0]);
        v[0][1] = x[r0];
        v[1][1] = x[r0 + 1];
    } else {
        // pairs of blocks side by side: words [column][block]
        tmem_get(tm + r0 * 8, v[0][0], v[0][1]);
#pragma unroll
        for (int a = G::WAIT_TMEM; a + 1 < G::R; a++) v[0][a] = ahead.w[a - G::WAIT_TMEM];
        const double2 w = buf[r0 * G::NT + tid];
        v[0][G::R - 1] = cpx{w.x, w.y};
    }
}
// ... and after them
template <class G>
__device__ __forceinline__ void enc_between(cpx (&v)[G::COLUMNS][G::R], const root_t *tab, uint32_t r0, uint32_t tid) {
#pragma unroll
    for (int i = 0; i < G::COLUMNS; i++) fft_outer_inverse<G::CL>(v[i], tab, tid, r0 + i);
}

// One block of a product waits for the last one.
template <class G>
__device__ __forceinline__ void enc_wait(const cpx (&x)[16], double2 *wait, uint32_t tm, uint32_t b, uint32_t tid) {
    if (G::WAIT_TMEM > 0 && (int)b < G::WAIT_TMEM) {
        if constexpr (G::R > 2) {
#pragma unroll
            for (int r = 0; r < 16; r++) {
                asm volatile("tcgen05.st.sync.aligned.32x32b.x4.b32 [%0], {%1, %2, %3, %4};" ::"r"(tm + r * 8 + b * 4),
                             "r"(__double2loint(x[r].re)), "r"(__double2hiint(x[r].re)), "r"(__double2loint(x[r].im)),
                             "r"(__double2hiint(x[r].im))
                             : "memory");
            }
        } else {
#pragma unroll
            for (int r = 0; r < 16; r += 2) tmem_put(tm + b * 64 + r * 4, x[r], x[r + 1]);
        }
        tmem_wait_put();
    } else {
        double2 *dst = wait + (b - G::WAIT_TMEM) * G::NB + tid;
#pragma unroll
        for (int r = 0; r < 16; r++) __stcg(dst + r * G::NT, make_double2(x[r].re, x[r].im));
    }
}

__device__ __forceinline__ int64_t fft_round(double z) { return fft_round_bits(z) - FFT_ROUND_BITS; }

// A low piece's values are parked for the same thread, which will join the top one.
template <class G>
__device__ __forceinline__ void enc_park(const cpx (&v)[G::COLUMNS][G::R], unsigned char *park, uint32_t tm, bool narrow,
                                         uint32_t r0, uint32_t tid) {
    const uint32_t i0 = r0 * G::R * 2;
    if (G::ALL_NARROW || narrow) {
        uint32_t w[G::K];
#pragma unroll
        for (int i = 0; i < G::K; i++) {
            const cpx &c = v[i / (2 * G::R)][(i / 2) % G::R];
            w[i] = (uint32_t)fft_round_bits((i & 1) ? c.im : c.re);
        }
        if constexpr (G::PARK_TMEM) {
            static_assert(G::K == 8, "eight words at a time");
            tmem_put8(tm + G::PARK_AT + i0, w);
        } else {
#pragma unroll
            for (int i = 0; i < G::K; i += 4)
                __stcg(reinterpret_cast<uint4 *>(park) + (i0 + i) / 4 * G::NT + tid, make_uint4(w[i], w[i + 1], w[i + 2], w[i + 3]));
        }
    } else {                                              // two pieces, 61 bits on the longer rings
        long long *p = reinterpret_cast<long long *>(park) + i0 * G::NT + tid;
#pragma unroll
        for (int i = 0; i < G::K; i++) {
            const cpx &c = v[i / (2 * G::R)][(i / 2) % G::R];
            __stcg(p + i * G::NT, (long long)fft_round((i & 1) ? c.im : c.re));
        }
    }
}
template <class G>
__device__ __forceinline__ void enc_parked(int64_t (&val)[G::K], const unsigned char *park, const EncAhead<G> &ahead, uint32_t tm,
                                           bool narrow, uint32_t joins, uint32_t r0, uint32_t tid) {
    const uint32_t i0 = r0 * G::R * 2;
    // the low piece's product: the word itself, or, of a pair, its lower 16 bits (signed) or what they leave
    auto low_of = [&](int w) {
        if (joins < 2) return w;
        return joins == 2 ? (int)(int16_t)w : (w - (int)(int16_t)w) >> 16;
    };
    if (joins == 0) return;
    if (G::ALL_NARROW || narrow) {
        if constexpr (G::PARK_TMEM) {
            uint32_t w[8];
            tmem_get8(tm + G::PARK_AT + i0, w);
#pragma unroll
            for (int i = 0; i < G::K; i++) val[i] += low_of((int)w[i]);
        } else {
#pragma unroll
            for (int i = 0; i < G::K; i++) val[i] += low_of(ahead.low[i]);
        }
    } else {
#pragma unroll
        for (int i = 0; i < G::K; i++) val[i] += __ldcg(reinterpret_cast<const long long *>(park) + (i0 + i) * G::NT + tid);
    }
}

// One of the ITEMS of a ciphertext's random draws, by a thread block: first those of e0, then e1, then u.
template <int CL>
__device__ __forceinline__ void enc_sample_item(const GaussTables &gt, uint32_t part, uint64_t seed, uint32_t t, uint32_t client,
                                                unsigned char *samples) {
    using G = EncRing<CL>;
    constexpr uint32_t NB = G::NB, NT = G::NT, R = G::R, n = G::n;
    if (part < 2 * G::E_ITEMS) {
        const uint32_t second = part >= G::E_ITEMS ? 1 : 0, b = (part - second * G::E_ITEMS) * 2 * NT + threadIdx.x;
        int2 e[2];
        gauss_pairs<2>(e, gt, seed, b, NT, t, client, second ? TAG_ENC_E1 : TAG_ENC_E0);
        char2 *dst = reinterpret_cast<char2 *>(samples + (second ? G::E1 : G::E0));
#pragma unroll
        for (int j = 0; j < 2; j++) __stcg(dst + b + j * NT, make_char2((signed char)e[j].x, (signed char)e[j].y));
    } else {
        // four columns of one half, all their rows
#pragma unroll
        for (uint32_t j = 0; j < G::U_COLUMNS; j++) {
            const uint32_t w = ((part - 2 * G::E_ITEMS) * G::U_COLUMNS + j) * NT + threadIdx.x;
            uint32_t f[4] = {0, 0, 0, 0};
#pragma unroll
            for (uint32_t a = 0; a < R; a++) {
                const u32x4 v = stream_block(seed, (w / (NB / 4)) * (n / 4) + a * (NB / 4) + w % (NB / 4), t, client, TAG_ENC_U);
                f[0] |= (uint32_t)(ternary_from_word(v.x) + 1) << (2 * a);
                f[1] |= (uint32_t)(ternary_from_word(v.y) + 1) << (2 * a);
                f[2] |= (uint32_t)(ternary_from_word(v.z) + 1) << (2 * a);
                f[3] |= (uint32_t)(ternary_from_word(v.w) + 1) << (2 * a);
            }
            unsigned char *dst = samples + G::U;
            if constexpr (R <= 4) __stcg(reinterpret_cast<uint32_t *>(dst) + w, f[0] | f[1] << 8 | f[2] << 16 | f[3] << 24);
            else __stcg(reinterpret_cast<uint2 *>(dst) + w, make_uint2(f[0] | f[1] << 16, f[2] | f[3] << 16));
        }
    }
}

// Every S-th of `count` items from the first one on, leaving out those of e0 or e1 from `skip` on.  Not inlined: the samplers' registers would
// cost the kernel that calls it spills.  The tables go where the transforms will work: 3 KB more shared memory to a block would leave the SM
// 28 KB of L1 instead of 60 (N = 32768, 200 ciphertexts: 784 -> 816 us).
template <int CL>
__device__ __noinline__ void enc_sample_items(const void *gauss, GaussTables &gt, uint32_t first, uint32_t S, uint32_t count, uint32_t skip, uint64_t seed,
                                              uint32_t t, uint32_t client, unsigned char *samples) {
    __syncthreads();                                      // the buffer's last readers are done
    gauss_tables_load(gt, gauss, threadIdx.x, FftLay::NT);
    __syncthreads();
#pragma unroll 1
    for (uint32_t i = first; i < count; i += S) enc_sample_item<CL>(gt, i < skip ? i : i + EncRing<CL>::E_ITEMS, seed, t, client, samples);
}

// The random draws of T ciphertexts from number t0 on, [T][SAMPLES], for the kernel below.  Drawn there, by clusters that have 16
// warps to an SM and nothing else to do meanwhile, they take 15 % of the time; here the integer multiplies of Philox set it.
// That kernel may start when every thread block of this one has: it waits for the end of this one where it needs the samples.
template <int CL>
__global__ void __launch_bounds__(FftLay::NT)
enc_sample_kernel(const void *gauss, EncDraw draw, uint32_t T, unsigned char *samples) {
    using G = EncRing<CL>;
    __shared__ GaussTables gt;
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    gauss_tables_load(gt, gauss, threadIdx.x, G::NT);
    __syncthreads();
#pragma unroll 1
    for (uint32_t i = blockIdx.x; i < T * G::ITEMS; i += gridDim.x) {
        const uint32_t tl = i / G::ITEMS;
        enc_sample_item<CL>(gt, i % G::ITEMS, draw.seed, draw.t0 + tl, draw.client, samples + (size_t)tl * G::SAMPLES);
    }
}

// A cluster of thread blocks encrypts ciphertexts one after the other: first it prepares one together -- u
// is transformed, the slots are encoded and e0 added, in R blocks
// of 2^12 points that its thread blocks share out -- and then each of them works off its own units
// (component, limb) of it: per piece of the key and block of the transform the product with the key's table
// and the inverse transform, per piece the stages between blocks and the rounding, then joining, error and
// message terms, canonical residues.  HBM sees the slots and the ciphertext once, the cluster meets twice
// per ciphertext.  (With the blocks of every product spread over the cluster it met twice per
// piece, and waiting for one another took 6, 9 and 11 of 19, 22 and 26 thousand clocks per block and piece for R = 2, 4, 8.)
//
// Two thread blocks fit on an SM on every ring, so that one's memory phases meet the other's arithmetic.
// The clusters fetch ciphertexts as they finish (with equal shares dealt out beforehand the slowest took 16 %
// longer than the mean).  Of the `rem` ciphertexts after the last whole round each is cut in `parts`: clusters that
// all prepare it and share its units.
//
// What bounds it: in the transforms shared memory (3360 of 3500 clocks a block of 2^12 points and SM: two exchanges of 1024, the key's table in and
// out 1024, twiddles 288), between them latency at the 16 warps that registers leave; the fp64 pipe is 36 to 41 % busy.  Measured, against
// modular transforms of every limb; with the draws of u and the errors by the clusters; and with these from the kernel above and what a
// product needs to know in shared memory:
//   N = 2^13, L = 3, 1 ciphertext       67.7 us -> 30.7 us -> 23.5 us
//   N = 2^14, L = 4, 313 ciphertexts    0.69 ms -> 0.32 ms -> 0.30 ms
//   N = 2^14, L = 4, 1429 ciphertexts   2.82 ms -> 1.38 ms -> 1.27 ms (1.2 TB/s of ciphertext)
//   N = 2^15, L = 6, 672 ciphertexts              2.69 ms -> 2.33 ms (0.9 TB/s)
//
struct EncTable { const EncJobs *jobs; uint32_t products; };
// PAIRS: some units are of two limbs (the code for both kinds costs the others 1.5 %).
template <int CL, bool PAIRS>
__global__ void __launch_bounds__(FftLay::NT, 2)
encrypt_fft_kernel(const __grid_constant__ CtxDev c, const __grid_constant__ EncTable made, const KeysDev k, const float *sel,
                   const EncDraw draw, unsigned char *samples, unsigned char *work, uint64_t *ct, uint32_t T, uint32_t S, uint32_t most_parts) {
    using G = EncRing<CL>;
    constexpr uint32_t N = G::N, n = G::n, NB = G::NB, NT = G::NT, R = G::R;
    extern __shared__ __align__(128) unsigned char smem[];
    double2 *buf = reinterpret_cast<double2 *>(smem);
    root_t *tab = reinterpret_cast<root_t *>(smem + (size_t)NB * 16);
    int8_t *e1_smem = reinterpret_cast<int8_t *>(tab + G::Tab::WORDS);
    __shared__ EncJobs jobs;
    __shared__ uint32_t tmem_base;
    __shared__ __align__(8) uint64_t key_bar;
    const uint32_t rank = blockIdx.x % S, cid = blockIdx.x / S, nc = gridDim.x / S;
    enc_jobs_load(jobs, made.jobs);
    for (uint32_t i = threadIdx.x; i < (uint32_t)G::Tab::WORDS; i += NT) tab[i] = c.fft_inv[i];
    if (threadIdx.x == 0) {
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"((uint32_t)__cvta_generic_to_shared(&key_bar)) : "memory");
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    CopyTurns turns(KEY_TRIES);
    const uint32_t tm = tmem_take(&tmem_base);            // and the tables are there
    unsigned char *common = work + (size_t)cid * (G::SHARED + S * G::OWN), *own = common + G::SHARED + rank * G::OWN;
    double2 *uhat = reinterpret_cast<double2 *>(common);                        // [R][16][NT]
    // message and e0 by residue of the coefficient's number, as the encoder's blocks leave them: [2 halves][R][NB],
    // coefficient R kk + b at kk of row b
    long long *terms = reinterpret_cast<long long *>(common + G::UHAT);
    auto term_of = [&](uint32_t coef) {
        return terms + ((coef & (n - 1)) >> CL) + ((coef & (R - 1)) + (coef >= n ? R : 0)) * NB;
    };
    uint32_t *flags = reinterpret_cast<uint32_t *>(terms + N);
    double2 *wait = reinterpret_cast<double2 *>(own);
    unsigned char *park = own + G::WAIT;
    auto meet = [&]() {                                   // everything the cluster wrote is visible to all of it
        if (S > 1) {
            asm volatile("barrier.cluster.arrive.release;" ::: "memory");
            asm volatile("barrier.cluster.wait.acquire;" ::: "memory");
        } else {
            __syncthreads();
        }
    };

    const uint32_t whole = T / nc * nc, rem = T - whole;
    const uint32_t parts = rem ? (nc / rem < most_parts ? nc / rem : most_parts) : 1;
    const uint32_t items = whole + rem * parts;           // at least as many as clusters
    const uint32_t products = made.products, all = 2 * products;
    const bool leader = rank == 0 && threadIdx.x == 0;
    uint32_t next_item = cid;
    asm volatile("griddepcontrol.wait;" ::: "memory");    // for samples drawn by the kernel above
#pragma unroll 1
    for (uint32_t it = 0; next_item < items; it++) {
        const uint32_t item = next_item;
        // words of two turns: a word is written again after the others have read it and met
        if (leader) {
            __stcg(flags + (it & 1u), 0u);
            __stcg(flags + 2 + (it & 1u), nc + atomicAdd(c.deal, 1u));
        }
        uint32_t tl = item, part = 0, of = 1;
        if (item >= whole) {
            tl = whole + (item - whole) / parts;
            part = (item - whole) % parts;
            of = parts;
        }
        const uint32_t first = jobs.start[all * part / of], last = jobs.start[all * (part + 1) / of];
        const uint32_t job_end = jobs.start[all * (part * S + rank + 1) / (of * S)];
        uint32_t job = jobs.start[all * (part * S + rank) / (of * S)];
        const bool c0_too = first < products, c1_too = last > products;
        unsigned char *drawn = samples + (size_t)tl * G::SAMPLES;

        if (draw.inside && first != last) {
            // clusters that share a ciphertext write the same samples
            constexpr uint32_t E = G::E_ITEMS;
            const uint32_t count = G::ITEMS - (c0_too && c1_too ? 0 : E);
            enc_sample_items<CL>(c.gauss, *reinterpret_cast<GaussTables *>(smem), rank, S, count, c0_too ? (c1_too ? G::ITEMS : E) : 0, draw.seed, draw.t0 + tl, draw.client, drawn);
        }
        meet();                                           // the samples are there, and nobody works on the last ciphertext any more
        next_item = __ldcg(flags + 2 + (it & 1u));
        if (first == last) continue;                      // more parts than units
        // ---- preparation: the transform of u and the encoder's network, 2 R blocks of 2^12 points ----
        int far = 0;
#pragma unroll 1
        for (uint32_t item = rank; item < 2 * R; item += S) {
            const uint32_t b = item & (R - 1);
            if (item < R) {
                cpx x[16];
                {
                    const OuterPath<CL> outer(c.fft_fwd, b);
                    const typename G::Row *p = reinterpret_cast<const typename G::Row *>(drawn + G::U) + fresh_tid();     // [2 halves][NB]
                    auto ternary = [](uint32_t f) {       // 0, 1, 2 -> -1.0, 0.0, 1.0
                        return __hiloint2double(f == 1 ? 0 : 0x3ff00000 | (int)((f == 0 ? 1u : 0u) << 31), 0);
                    };
#pragma unroll
                    for (int r = 0; r < 16; r++) {
                        const uint32_t re = __ldcg(p + NT * r), im = __ldcg(p + NB + NT * r);
                        cpx z[R];
#pragma unroll
                        for (uint32_t a = 0; a < R; a++) z[a] = cpx{ternary((re >> (2 * a)) & 3u), ternary((im >> (2 * a)) & 3u)};
                        x[r] = outer.apply(z);
                    }
                }
                fft_forward<CL, true>(x, buf, c.fft_fwd, b, fresh_tid());
                double2 *dst = uhat + b * NB + fresh_tid();
#pragma unroll
                for (int r = 0; r < 16; r++) __stcg(dst + r * NT, make_double2(x[r].re, x[r].im));
            } else if (c0_too) {
                const float *slots = sel + (size_t)tl * n;
                const uint32_t first_of_row = CL ? bitrev(b, CL ? CL : 1) : 0u;
                long long *row = terms + first_of_row * NB;
                const int8_t *e0 = reinterpret_cast<const int8_t *>(drawn + G::E0) + first_of_row;
                __syncthreads();                          // the buffer's last readers are done
                if (encode_block_in_place<Lay<FftLay::LB, 4>>(
                        c, [&](uint32_t i) { return encoder_stages<CL>(slots, c.ftw, n, b, i); },
                        reinterpret_cast<uint64_t *>(buf), CL,
                        [&](uint32_t kk) { return make_char2(__ldcg(e0 + R * kk), __ldcg(e0 + n + R * kk)); },
                        [&](uint32_t kk, int64_t re, int64_t im, char2 e) {
                            re += e.x;
                            im += e.y;
                            far |= (re < 0 ? -re : re) >= c.term_limit || (im < 0 ? -im : im) >= c.term_limit;
                            __stcg(row + kk, (long long)re);
                            __stcg(row + R * NB + kk, (long long)im);
                        }))
                    atomicOr(c.status, STATUS_RANGE);
            }
        }
        if (far) atomicOr(flags + (it & 1u), 1u);         // a term of c0 needs reducing first
        meet();
        if (job == job_end) continue;
        const bool big = __ldcg(flags + (it & 1u)) != 0;
        const int8_t *e1 = reinterpret_cast<const int8_t *>(drawn + G::E1);
        if constexpr (G::E_IN_SMEM) {
            if (c1_too) {
                for (uint32_t i = threadIdx.x; i < N / 16; i += NT)
                    reinterpret_cast<uint4 *>(e1_smem)[i] = __ldcg(reinterpret_cast<const uint4 *>(e1) + i);
                __syncthreads();
            }
        }
        const int8_t *e1_at = G::E_IN_SMEM ? e1_smem : e1;
        if constexpr (R == 1) {
            const double2 *uh = uhat + fresh_tid();
#pragma unroll
            for (int r = 0; r < 16; r += 2) {
                const double2 a = __ldcg(uh + r * NT), b = __ldcg(uh + (r + 1) * NT);
                tmem_put(tm + r * 4, cpx{a.x, a.y}, cpx{b.x, b.y});
            }
            tmem_wait_put();
        }

        // ---- this block's units ----
        auto wait_for_key = [&]() {
            if (!turns.take([&](uint32_t parity) { return key_try(&key_bar, parity); })) atomicOr(c.status, STATUS_COPY);
        };
        auto key_of = [&](uint32_t i, uint32_t b) {
            const uint32_t comp = i >= products ? 1 : 0;
            return k.fft_pk + (size_t)(jobs.job[i - comp * products].key[comp] + b) * NB;
        };
        if constexpr (!(G::E_IN_SMEM)) __syncthreads();   // the buffer's last readers are done
        if (threadIdx.x == 0 && !turns.lost()) key_fetch(buf, key_of(job, 0), &key_bar);
#pragma unroll 1
        for (; job < job_end; job++) {
            const uint32_t comp = job >= products ? 1 : 0;
            const EncJob &e = jobs.job[job - comp * products];
#pragma unroll 1
            for (uint32_t b = 0; b < R; b++) {
                cpx x[16];
                {
                    const uint32_t tid = fresh_tid();
                    const double2 *key = buf + tid;
                    if constexpr (R == 1) {
                        wait_for_key();
#pragma unroll
                        for (int h = 0; h < 2; h++) {
                            uint32_t w[32];
                            tmem_get32(tm + h * 32, w);
#pragma unroll
                            for (int r = 0; r < 8; r++)
                                x[8 * h + r] = cpx_mul(tmem_cpx(w + 4 * r), key[(8 * h + r) * NT].x, key[(8 * h + r) * NT].y);
                        }
                    } else {
                        const double2 *uh = uhat + b * NB + tid;
#pragma unroll
                        for (int r = 0; r < 16; r++) {
                            const double2 w = __ldcg(uh + r * NT);
                            x[r] = cpx{w.x, w.y};
                        }
                        wait_for_key();
#pragma unroll
                        for (int r = 0; r < 16; r++) x[r] = cpx_mul(x[r], key[r * NT].x, key[r * NT].y);
                    }
                }
                // the next key may come as soon as the buffer is read; where a column loop needs the buffer, after it
                const bool more = b + 1 < R || job + 1 < job_end;
                auto fetch_next = [&]() {
                    __syncthreads();
                    if (more && threadIdx.x == 0 && !turns.lost())
                        key_fetch(buf, b + 1 < R ? key_of(job, b + 1) : key_of(job + 1, 0), &key_bar);
                };
                fft_inverse<0>(x, buf, tab, fresh_tid(), [&] {
                    if (R <= 2 || b + 1 < R) fetch_next();
                });
                const uint32_t tid = fresh_tid();
                if (b + 1 < R) {
                    enc_wait<G>(x, wait, tm, b, tid);
                    continue;
                }
                if constexpr (R > 2) {
                    // the thread's own words: the columns are finished in a loop, which registers do not allow
#pragma unroll
                    for (int r = 0; r < 16; r++) buf[r * NT + tid] = make_double2(x[r].re, x[r].im);
                }
                constexpr int K = G::K;
                const uint32_t what = e.what, joins = what >> EncJob::JOINS;
                const bool narrow = (what & EncJob::NARROW) != 0;
                EncAhead<G> ahead;
                if constexpr (G::FAR_AHEAD) ahead.fetch_wait(wait, 0, tid);
                if (what & EncJob::PARKS) {
#pragma unroll(R <= 2 ? 16 : 1)
                    for (uint32_t r0 = 0; r0 < 16; r0 += G::COLUMNS) {
                        cpx v[G::COLUMNS][R];
                        if constexpr (!G::FAR_AHEAD) ahead.fetch_wait(wait, r0, tid);
                        enc_columns<G>(v, x, buf, ahead, tm, r0, tid);
                        if (G::FAR_AHEAD && r0 + G::COLUMNS < 16) ahead.fetch_wait(wait, r0 + G::COLUMNS, tid);
                        enc_between<G>(v, tab, r0, tid);
                        enc_park<G>(v, park, tm, narrow, r0, tid);
                    }
                    if constexpr (G::PARK_TMEM) tmem_wait_put();
                    if constexpr (R > 2) fetch_next();
                    continue;
                }
                const uint32_t j = what & (EncJob::PARKS - 1);
                const uint64_t q = e.q;
                uint64_t *out = ct + (((size_t)tl * 2 + comp) * c.L + j) * N + tid;
                const FftJoin join(q, e.scale, e.shift);
                // the offsets of a thread's coefficients are multiples of R, so they split off the number of the first
                const long long *my_terms = term_of(tid);
                auto terms_of = [&](int64_t (&val)[K], uint32_t r0) {
                    if (comp == 1) {
#pragma unroll
                        for (int i = 0; i < K; i++) val[i] = e1_at[enc_coefficient<G>(r0, i) + tid];
                    } else {
#pragma unroll
                        for (int i = 0; i < K; i++) {
                            const uint32_t at = enc_coefficient<G>(r0, i);
                            val[i] = __ldcg(my_terms + ((at & (n - 1)) >> CL) + (at >= n ? R * NB : 0));
                        }
                    }
                };
                int64_t next[K];
                terms_of(next, 0);
                if (G::FAR_AHEAD && joins && narrow) ahead.fetch_low(park, 0, tid);
#pragma unroll(R <= 2 ? 16 : 1)
                for (uint32_t r0 = 0; r0 < 16; r0 += G::COLUMNS) {
                    int64_t val[K];
#pragma unroll
                    for (int i = 0; i < K; i++) val[i] = big && comp == 0 ? 0 : next[i];
                    if (!G::FAR_AHEAD) {
                        if (r0 + G::COLUMNS < 16) terms_of(next, r0 + G::COLUMNS);
                        if (joins && narrow) ahead.fetch_low(park, r0, tid);
                    }
                    enc_parked<G>(val, park, ahead, tm, narrow, PAIRS || joins == 0 ? joins : 1, r0, tid);
                    cpx v[G::COLUMNS][R];
                    if (!G::FAR_AHEAD) ahead.fetch_wait(wait, r0, tid);
                    enc_columns<G>(v, x, buf, ahead, tm, r0, tid);
                    if (G::FAR_AHEAD && r0 + G::COLUMNS < 16) {
                        terms_of(next, r0 + G::COLUMNS);
                        if (joins && narrow) ahead.fetch_low(park, r0 + G::COLUMNS, tid);
                        ahead.fetch_wait(wait, r0 + G::COLUMNS, tid);
                    }
                    enc_between<G>(v, tab, r0, tid);
                    // streaming stores: the finished ciphertext should not push tables and scratch out of L2
#pragma unroll
                    for (int i = 0; i < K; i++) {
                        const cpx &w = v[i / (2 * (int)R)][(i / 2) % (int)R];
                        __stcs(reinterpret_cast<unsigned long long *>(out + enc_coefficient<G>(r0, i)),
                               (unsigned long long)fft_canonical(join(val[i], (i & 1) ? w.im : w.re), q));
                    }
                }
                if constexpr (R > 2) fetch_next();
                if (big && comp == 0) {
                    // terms beyond a quarter of the smallest prime: encoded updates are far below, so this is rare
                    const uint64_t mu = c.limb[j].mu;
#pragma unroll 1
                    for (uint32_t at = 0; at < N; at += NT)
                        out[at] = addmod(out[at], signed_residue(__ldcg(term_of(at + tid)), q, mu), q);
                }
            }
        }
    }
    if (threadIdx.x == 0 && turns.lost())                 // that copy may still be on its way into this block's memory
        for (uint32_t i = 0; i < KEY_TRIES && !key_try(&key_bar, turns.parity()); i++) {}
    if (leader && atomicAdd(c.deal + 1, 1u) + 1 == nc) {  // the last cluster leaves the words as it found them
        c.deal[0] = 0;
        c.deal[1] = 0;
    }
    tmem_give(tmem_base);
}

// ===========================================================================
// decryption + decoding:  d = c0 + c1 s on limb 0, centred, then the slot transform
// ===========================================================================

// a double from a 32-bit integer: the integer plus 2^31 as the low word of 2^52 + ...
__device__ __forceinline__ double fft_from_int32(int v) {
    return f64_sub(__hiloint2double(0x43300000, (int)((uint32_t)v ^ 0x80000000u)), 4503601774854144.0);      // 2^52 + 2^31
}

// A cluster decrypts and decodes a range of ciphertexts: per piece of c1 a forward
// transform, the product with the transformed secret, an inverse transform; joining, c0, centring;
// then the slot transform, which is the forward transform again (a slot is the value at one of the
// roots; `slot_of` puts the values in order through shared memory).  Only the two limb-0
// polynomials are read and the n decoded values written.
//
// c0 and the joined lower pieces wait in tensor memory, in the words of the threads that will join them; c1 is read
// by all its loads at once, and cut in 32-bit arithmetic if its pieces are two.  (Reading eight values at a time from L2
// and cutting in 64 bits, loading and joining took 28 of 65 thousand clocks per ciphertext of N = 8192.)
//
// Bound by its chain of transforms, exchanges and loads on few ciphertexts: 68 of N = 2^15 take 141 us by modular transforms in
// separate kernels and 84 us here.
template <int CL>
__global__ void __launch_bounds__(FftLay::NT, 2)
decrypt_fft_kernel(const __grid_constant__ CtxDev c, const KeysDev k, const uint64_t *ct, uint32_t level,
                   double *z, uint32_t T) {
    using G = FftRing<CL>;
    constexpr uint32_t n = G::n, NB = G::NB, NT = G::NT, R = G::R;
    constexpr size_t N = G::N;
    extern __shared__ __align__(128) unsigned char smem[];
    double2 *buf = reinterpret_cast<double2 *>(smem);
    root_t *tab = reinterpret_cast<root_t *>(smem + (size_t)NB * 16);
    __shared__ uint32_t tmem_base;
    const uint32_t rank = blockIdx.x % R, cid = blockIdx.x / R, nc = gridDim.x / R;
    for (uint32_t i = threadIdx.x; i < (uint32_t)G::Tab::WORDS; i += NT) tab[i] = c.fft_inv[i];
    buffer_free<CL>();
    const uint32_t tm = tmem_take(&tmem_base);            // and the tables are there
    constexpr uint32_t C0_AT = 0, PARK_AT = 64;           // 32 values of two words each
    const FftSplit &f = c.dec_split;
    const uint64_t q = c.limb[0].q;
    const int64_t half_q = (int64_t)(q / 2);
    const double inv_delta = __longlong_as_double((long long)(1023 - c.log2_delta) << 52);
    const uint32_t t_end = (uint32_t)((uint64_t)T * (cid + 1) / nc);
    auto centred = [&](uint64_t v) { return v > (uint64_t)half_q ? (int64_t)(v - q) : (int64_t)v; };
    auto get4 = [&](uint32_t at, int64_t (&v)[4]) {
        uint32_t w[8];
        tmem_get8(tm + at, w);
#pragma unroll
        for (int i = 0; i < 4; i++) v[i] = (int64_t)(((uint64_t)w[2 * i + 1] << 32) | w[2 * i]);
    };
    auto put4 = [&](uint32_t at, const int64_t (&v)[4]) {
        const uint32_t w[8] = {(uint32_t)v[0], (uint32_t)((uint64_t)v[0] >> 32), (uint32_t)v[1], (uint32_t)((uint64_t)v[1] >> 32),
                               (uint32_t)v[2], (uint32_t)((uint64_t)v[2] >> 32), (uint32_t)v[3], (uint32_t)((uint64_t)v[3] >> 32)};
        tmem_put8(tm + at, w);
    };
#pragma unroll 1
    for (uint32_t t = (uint32_t)((uint64_t)T * cid / nc); t < t_end; t++) {
        const uint64_t *c0 = ct + ((size_t)t * 2 * level) * N, *c1 = c0 + level * N;
        cpx x[16];
        // the pieces, then the slot transform as one more turn of the same code
#pragma unroll 1
        for (uint32_t p = 0; p <= f.pieces; p++) {
            if (p < f.pieces) {
                const uint64_t *src = c1 + fresh_tid();
                uint64_t raw[32];
#pragma unroll
                for (int i = 0; i < 32; i++) raw[i] = __ldg(src + fft_coefficient<G>(i, rank));
                if (f.pieces == 2) {
                    const uint32_t w = f.shift[1];                       // at most 30
                    if (p == 0) {
#pragma unroll
                        for (int o = 0; o < 16; o++) {
                            const uint32_t re = (uint32_t)centred(raw[2 * o]), im = (uint32_t)centred(raw[2 * o + 1]);
                            x[o] = cpx{fft_from_int32((int)(re << (32 - w)) >> (32 - w)), fft_from_int32((int)(im << (32 - w)) >> (32 - w))};
                        }
                    } else {
                        const int64_t round = (int64_t)1 << (w - 1);
#pragma unroll
                        for (int o = 0; o < 16; o++)
                            x[o] = cpx{fft_from_int32((int)((centred(raw[2 * o]) + round) >> w)),
                                       fft_from_int32((int)((centred(raw[2 * o + 1]) + round) >> w))};
                    }
                } else {
#pragma unroll
                    for (int o = 0; o < 16; o++)
                        x[o] = cpx{fft_from_int(fft_piece(f, centred(raw[2 * o]), p)), fft_from_int(fft_piece(f, centred(raw[2 * o + 1]), p))};
                }
            }
            fft_spread<G>(x, buf, c.fft_fwd, rank, fresh_tid());
            fft_forward<CL>(x, buf, c.fft_fwd, rank, fresh_tid());
            if (p == f.pieces) break;
            {
                const double2 *key = k.fft_s + (size_t)rank * NB + fresh_tid();
#pragma unroll
                for (int r = 0; r < 16; r++) {
                    const double2 w = load_passing(key + r * NT);
                    x[r] = cpx_mul(x[r], w.x, w.y);
                }
            }
            fft_inverse<CL>(x, buf, tab, fresh_tid());
            fft_gather<G>(x, buf, tab, rank, fresh_tid());
            if (p + 1 < f.pieces) {
                const uint32_t sh = f.shift[p];
#pragma unroll
                for (int i0 = 0; i0 < 32; i0 += 4) {
                    int64_t v[4];
                    if (p) get4(PARK_AT + 2 * i0, v);
#pragma unroll
                    for (int i = 0; i < 4; i++) {
                        const int64_t low = fft_round((i & 1) ? x[(i0 + i) >> 1].im : x[(i0 + i) >> 1].re) << sh;
                        v[i] = p ? v[i] + low : low;
                    }
                    put4(PARK_AT + 2 * i0, v);
                }
                if (p + 2 == f.pieces) {
                    // c0, while nothing else is wanted of the registers
                    const uint64_t *src = c0 + fresh_tid();
                    uint64_t raw[32];
#pragma unroll
                    for (int i = 0; i < 32; i++) raw[i] = __ldg(src + fft_coefficient<G>(i, rank));
#pragma unroll
                    for (int i0 = 0; i0 < 32; i0 += 4) {
                        const int64_t v[4] = {centred(raw[i0]), centred(raw[i0 + 1]), centred(raw[i0 + 2]), centred(raw[i0 + 3])};
                        put4(C0_AT + 2 * i0, v);
                    }
                }
                tmem_wait_put();
                continue;
            }
            const FftJoin join(f, q);
            const uint64_t *src = c0 + fresh_tid();
#pragma unroll
            for (int i0 = 0; i0 < 32; i0 += 4) {
                int64_t add[4], low[4] = {0, 0, 0, 0};
                if (f.pieces > 1) {
                    get4(C0_AT + 2 * i0, add);
                    get4(PARK_AT + 2 * i0, low);
                } else {
#pragma unroll
                    for (int i = 0; i < 4; i++) add[i] = centred(__ldg(src + fft_coefficient<G>(i0 + i, rank)));
                }
#pragma unroll
                for (int i = 0; i < 4; i++) {
                    cpx &w = x[(i0 + i) >> 1];
                    // |the product| <= q / 2 and a little, |c0| <= q / 2
                    int64_t d = join(low[i] + add[i], (i & 1) ? w.im : w.re);
                    if (d > half_q) d -= (int64_t)q;
                    else if (d < -half_q) d += (int64_t)q;
                    ((i & 1) ? w.im : w.re) = __ll2double_rn(d) * inv_delta;
                }
            }
        }
        // the slots of this block have one residue mod R: in order through the buffer
        const uint32_t tid = fresh_tid();
        double *order = reinterpret_cast<double *>(buf);
        const uint32_t *slot = c.slot_of + (size_t)rank * NB + tid;
        buffer_wait<CL>();
#pragma unroll
        for (int r = 0; r < 16; r++) order[__ldg(slot + r * NT) >> CL] = x[r].re;
        __syncthreads();
        double *zt = z + (size_t)t * n + (__ldg(c.slot_of + (size_t)rank * NB) & (R - 1));
#pragma unroll
        for (int r = 0; r < 16; r++) zt[(size_t)(tid + NT * r) << CL] = order[tid + NT * r];
        buffer_free<CL>();
    }
    buffer_wait<CL>();
    tmem_give(tmem_base);
}

// ---- launch --------------------------------------------------------------------------

#define FEDHE_FOR_RING(c, FN, ...)                          \
    switch ((c).logN) {                                     \
    case 13: return FN<0>(__VA_ARGS__);                     \
    case 14: return FN<1>(__VA_ARGS__);                     \
    case 15: return FN<2>(__VA_ARGS__);                     \
    default: return FN<3>(__VA_ARGS__);                     \
    }

// ---- how residues are cut -----------------------------------------------------------

static int bits_of(uint64_t q) {
    int bits = 0;
    while (q >> bits) bits++;
    return bits;
}
// the top pieces `most` bits wide, the lowest with what remains; narrow_bits: widest low piece whose product fits 32 bits
static void cut_residues(uint64_t q, int most, int narrow_bits, FftSplit &f) {
    const int bits = bits_of(q);
    f.pieces = (uint32_t)((bits + most - 1) / most);
    for (uint32_t p = 0; p < FFT_MAX_PIECES; p++) f.shift[p] = p && p < f.pieces ? (uint32_t)(bits - most * (int)(f.pieces - p)) : 0;
    f.narrow = f.pieces == 2 && (int)f.shift[1] <= narrow_bits;
    f.top_scale = ldexp(1.0, (int)f.shift[f.pieces - 1]) / (double)q;
}
// Decryption cuts for any c1.  Of the public key's limbs, if they go in pairs, two whose low pieces have products of 16 bits (up to 6 bits wide
// for N = 2^15, at 12 standard deviations: under 2^-102 a coefficient) share one product for both: three instead of
// four, for instance for primes of 45 bits.  Another limb of two pieces is cut as low as the low piece's product is sure
// to fit 32 bits (a coefficient is below N 2^(width - 1)), or else as high as the top one may be wide, where it
// fits all the same (exponent 95: under 2^-136).
// False for a prime that the kernels are not made for: more than two pieces, or, for N <= 2^14, a wide low one.
static bool cut_limbs(CtxDev &c, bool in_pairs, EncWay &w, EncJobs &jobs, size_t &words) {
    const int logN = (int)c.logN, sure = fft_sure_bits(logN), wide = fft_wide_bits(logN), narrow = fft_random_bits(logN, 32, FFT_NARROW_EXPONENT);
    uint32_t waiting = NO_LIMB;                        // unit of a limb that could share its low product
    w.units = 0;
    for (uint32_t j = 0; j < c.L; j++) {
        const uint64_t q = c.limb[j].q;
        const int bits = bits_of(q);
        const bool shares = in_pairs && bits > wide && bits - wide <= fft_random_bits(logN, 16, FFT_PAIR_EXPONENT);
        const bool low_fits = bits > wide && bits - sure + logN - 1 < 31;
        if (shares && waiting != NO_LIMB) {
            EncUnit &e = w.unit[waiting];
            cut_residues(c.limb[e.limb].q, wide, narrow, c.limb[e.limb].split[1]);
            cut_residues(q, wide, narrow, c.limb[j].split[1]);
            e.limb2 = j;
            e.products = 3;
            waiting = NO_LIMB;
            continue;
        }
        FftSplit &f = c.limb[j].split[in_pairs];
        cut_residues(q, low_fits ? sure : wide, narrow, f);
        w.unit[w.units] = EncUnit{j, NO_LIMB, f.pieces, 0};
        if (shares) waiting = w.units;
        w.units++;
    }
    for (uint32_t j = 0; j < c.L; j++) {
        const FftSplit &f = c.limb[j].split[in_pairs];
        if (f.pieces > 2 || (f.pieces == 2 && !f.narrow && logN <= 14)) return false;
    }
    w.products = 0;
    const uint32_t R = 1u << (logN - 13);
    for (uint32_t u = 0; u < w.units; u++) {
        EncUnit &e = w.unit[u];
        e.fft_key = words;
        for (uint32_t p = 0; p < e.products; p++) {
            const bool pair = e.limb2 != NO_LIMB, parks = pair ? p == 0 : p + 1 < e.products;
            const uint32_t j = pair && p == 2 ? e.limb2 : e.limb, joins = parks || e.products == 1 ? 0 : pair ? p + 1 : 1;
            const FftSplit &f = c.limb[j].split[in_pairs];
            EncJob &d = jobs.job[w.products + p];
            d.q = c.limb[j].q;
            d.scale = f.top_scale;
            for (uint32_t comp = 0; comp < 2; comp++) d.key[comp] = (uint32_t)(words / FftLay::NB) + (comp * e.products + p) * R;
            d.shift = f.shift[f.pieces - 1];
            d.what = j | (parks ? EncJob::PARKS : 0u) | (f.narrow ? EncJob::NARROW : 0u) | joins << EncJob::JOINS;
        }
        words += 2 * (size_t)e.products * (c.N / 2);
        w.products += e.products;
    }
    uint32_t begin = 0, of_unit = 0;
    for (uint32_t pos = 0; pos <= 2 * w.products; pos++) {
        if (pos > begin) begin += w.unit[of_unit++ % w.units].products;
        jobs.start[pos] = (uint8_t)begin;
    }
    return true;
}
bool fft_cut(CtxDev &c, EncWays &e) {
    cut_residues(c.limb[0].q, fft_sure_bits((int)c.logN), 31 - (int)c.logN, c.dec_split);
    c.term_limit = INT64_MAX;
    for (uint32_t j = 0; j < c.L; j++)
        if ((int64_t)(c.limb[j].q / 4) < c.term_limit) c.term_limit = (int64_t)(c.limb[j].q / 4);
    size_t words = 0;
    if (!cut_limbs(c, true, e.way[0], e.jobs[0], words)) return false;
    e.count = e.way[0].units < c.L ? 2 : 1;
    if (e.count == 1) words = 0;
    if (!cut_limbs(c, false, e.way[e.count - 1], e.jobs[e.count - 1], words)) return false;
    for (uint32_t i = 0; i < e.count; i++) {
        const EncWay &w = e.way[i];
        for (uint32_t of = 1; of < ENC_SHARES; of++) {
            uint32_t most = 0;
            for (uint32_t part = 0; part < of; part++) {
                const uint8_t *start = e.jobs[i].start;
                const uint32_t sum = start[2 * w.products * (part + 1) / of] - start[2 * w.products * part / of];
                most = sum > most ? sum : most;
            }
            e.most[i][of] = (uint16_t)most;
        }
    }
    return true;
}
static bool pairs_limbs(const CtxDev &c, uint32_t way) { return c.enc->way[way].units < c.L; }
size_t fft_key_words(const CtxDev &c) {
    size_t words = 0;
    for (uint32_t i = 0; i < c.enc->count; i++) words += 2 * (size_t)c.enc->way[i].products * (c.N / 2);
    return words;
}

// Asked how many thread blocks fit on an SM, the runtime answers 1 for any kernel that allocates tensor memory;
// two that take half of it each do run side by side.  This kernel has the same shape without it.
__global__ void __launch_bounds__(FftLay::NT, 2) enc_shape_kernel() {}

// shared memory that leaves no room for a second thread block on the SM, and the most that the kernel has besides the dynamic part
constexpr int ENC_ALONE_SMEM = 116 * 1024, ENC_STATIC_SMEM = 1280;
static_assert(sizeof(EncJobs) + 64 <= ENC_STATIC_SMEM, "static shared memory of the encryption");

// How many clusters of 1 .. ENC_MOST blocks the device holds at once, two blocks to an SM and one.
template <int CL>
static cudaError_t setup_ring(CtxDev &c, int n_sm) {
    using G = EncRing<CL>;
    static_assert(G::SMEM + ENC_STATIC_SMEM <= ENC_ALONE_SMEM - 3072, "two thread blocks to an SM");
    cudaError_t e;
    for (uint32_t i = 0; i < c.enc->count; i++)
        if ((e = cudaFuncSetAttribute(pairs_limbs(c, i) ? encrypt_fft_kernel<CL, true> : encrypt_fft_kernel<CL, false>,
                                      cudaFuncAttributeMaxDynamicSharedMemorySize, ENC_ALONE_SMEM)))
            return e;
    if ((e = cudaFuncSetAttribute(decrypt_fft_kernel<CL>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)FftRing<CL>::SMEM))) return e;
    if ((e = cudaFuncSetAttribute(enc_shape_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, ENC_ALONE_SMEM))) return e;
    for (uint32_t alone = 0; alone < 2; alone++)
        for (uint32_t S = 1; S <= ENC_MOST; S++) {
            cudaLaunchConfig_t cfg = {};
            cudaLaunchAttribute attr;
            cfg.blockDim = dim3(G::NT, 1, 1);
            cfg.gridDim = dim3(S, 1, 1);
            cfg.dynamicSmemBytes = alone ? ENC_ALONE_SMEM : G::SMEM + ENC_STATIC_SMEM;
            attr.id = cudaLaunchAttributeClusterDimension;
            attr.val.clusterDim.x = S;
            attr.val.clusterDim.y = 1;
            attr.val.clusterDim.z = 1;
            cfg.attrs = &attr;
            cfg.numAttrs = 1;
            int clusters = 0;
            if ((e = cudaOccupancyMaxActiveClusters(&clusters, enc_shape_kernel, &cfg))) return e;
            const int most = (alone ? 1 : 2) * n_sm / (int)S;
            c.enc_fit[alone][S] = (uint16_t)(clusters < most ? clusters : most);
        }
    return cudaSuccess;
}
static cudaError_t setup_this_ring(CtxDev &c, int n_sm) { FEDHE_FOR_RING(c, setup_ring, c, n_sm) }
cudaError_t fft_setup(CtxDev &c, int n_sm) {
    const cudaError_t e = setup_this_ring(c, n_sm);
    if (e) return e;
    c.sm_count = (uint32_t)n_sm;
    c.passes_most = passes_most(c);
    return cudaSuccess;
}

// The units' way, the thread blocks that work on a ciphertext together, whether they have their SMs to themselves, the
// clusters, and the clusters that may share a ciphertext of the last round.
struct EncPlan { uint32_t way, S, alone, clusters, parts; };

static EncPlan enc_plan_of(const CtxDev &c, uint32_t way, uint32_t S, uint32_t alone, uint32_t fit, uint32_t parts, size_t T) {
    const size_t each = fit / T < parts ? fit / T : parts;
    return EncPlan{way, S, alone, T >= fit ? fit : (uint32_t)(T * each), parts};
}

// With ciphertexts enough to fill the device: as many blocks as the ciphertext has of 2^12 points, or the next
// number below that shares its units out evenly.  With fewer, larger clusters, by these measurements (us, L = 3 or 4):
//   N = 8192, 25 ciphertexts: 1, 2, 3, 4, 8 blocks 79, 52, 43, 40, 43 (8 of them share SMs); 60: 2, 4 blocks 52, 55;
//     100: 1, 2 blocks 81, 72
//   N = 16384, 40: 2, 3, 6 blocks 110, 86, 75; 60: 2, 4 blocks 111, 92
// so the largest clusters that hold all ciphertexts at one block to an SM, if they can do the 2 R blocks of the
// preparation side by side, and else the largest that hold them at two.
static EncPlan enc_plan_by_size(const CtxDev &c, size_t T) {
    const uint32_t R = 1u << (c.logN - 13), units = 2 * c.enc->way[0].units, most = units < ENC_MOST ? units : ENC_MOST;
    uint32_t base = R < most ? R : most;
    while (units % base) base--;
    uint32_t S = base, one = 0, parts = (units + base - 1) / base;
    uint32_t alone = most, shared = most;
    while (alone > 1 && c.enc_fit[1][alone] < T) alone--;
    while (shared > base && c.enc_fit[0][shared] < T) shared--;
    if (c.enc_fit[1][alone] >= T && alone >= base && (alone >= 2 * R || alone == most)) S = alone, one = 1, parts = 1;
    else if (shared > base) S = shared, parts = 1;
    const uint32_t fit = c.enc_fit[one][S];
    // what is left after whole rounds of all clusters, or too few ciphertexts for the largest clusters: several to each
    if (S == most || T > fit) parts = (units + S - 1) / S;
    return enc_plan_of(c, 0, S, one, fit, parts, T);
}

// clusters that surely run at once: with sizes that do not divide the SMs of a part of the chip the last one may have to wait
static uint32_t enc_sure_fit(const CtxDev &c, uint32_t alone, uint32_t S) {
    const uint32_t fit = c.enc_fit[alone][S];
    return S > 2 && S < 8 && fit > 1 ? fit - 1 : fit;
}

// What a plan takes, in us: a round is fixed + by_size / S + product * (block transforms of the busiest block's products),
// fitted to 10,000 measurements of all plans for up to 200 ciphertexts of 2 to 12 limbs of 45 and 60 bits (nine of ten within
// 10 %), for two blocks to an SM and for one, when the clusters drew for themselves.  Not fitted again since: plans
// take 9 to 13 % less now at N = 16384 (4 limbs, 1 to 60 ciphertexts) and 32768 (6 limbs), 4 to 9 % at 65536 (2 limbs, 24 to 600), and where
// an estimate is compared with another path's (encrypt_by_passes) it is too high by that.
struct EncCost { double fixed, by_size, product; };
static const EncCost ENC_COST[4][2] = {{{27.3, 12.7, 7.7}, {33.1, 2.2, 4.9}},
                                       {{27.4, 40.1, 9.1}, {43.5, 13.7, 5.7}},
                                       {{-2.2, 160.6, 12.6}, {26.2, 76.9, 6.8}},
                                       {{-27.8, 410.0, 15.6}, {15.8, 226.7, 8.3}}};
static double enc_plan_us(const CtxDev &c, const EncPlan &p, size_t T) {
    const uint32_t ring = c.logN - 13;
    auto round = [&](uint32_t clusters, uint32_t parts) {
        const EncCost &k = ENC_COST[ring][p.alone || clusters <= enc_sure_fit(c, 1, p.S)];
        return k.fixed + k.by_size / p.S + k.product * (c.enc->most[p.way][p.S * parts] << ring);
    };
    const size_t whole = T / p.clusters;
    const uint32_t rem = (uint32_t)(T % p.clusters);
    double us = whole ? (double)whole * round(p.clusters, 1) : 0.0;
    if (rem) {
        const uint32_t parts = p.clusters / rem < p.parts ? p.clusters / rem : p.parts;
        us += round(rem * parts, parts);
    }
    return us;
}

// The plan by size, or for up to a round or two of ciphertexts of N = 16384 and up another one if it should be 5 % faster (10 % at N = 65536):
// clusters of 2, 4, 6 or 8, several of them to a ciphertext, and limbs by themselves.  Measured (us, by size and so; primes of 45 bits):
//   N = 16384, L = 2, 1 ciphertext 106, 81; L = 12, 9 of them 116, 68; L = 4, 74 of them 159, 102
//   N = 32768, L = 2, 1 of them 173, 101; L = 6, 9 of them 128, 92; L = 8, 36 of them 322, 236
static EncPlan enc_plan(const CtxDev &c, size_t T) {
    EncPlan best = enc_plan_by_size(c, T);
    const uint32_t R = 1u << (c.logN - 13);
    if (best.clusters < 1 || R == 1 || T > (R == 8 ? 1u : 2u) * c.enc_fit[0][R]) return best;
    double us = (R == 8 ? 0.9 : 0.95) * enc_plan_us(c, best, T);
    for (uint32_t way = 0; way < c.enc->count; way++)
        for (uint32_t S = 2; S <= ENC_MOST; S += 2)
            for (uint32_t alone = 0; alone < 2; alone++) {
                const uint32_t fit = enc_sure_fit(c, alone, S), units = 2 * c.enc->way[way].units;
                if (fit < 1) continue;
                const EncPlan p = enc_plan_of(c, way, S, alone, fit, (units + S - 1) / S, T);
                const double t = enc_plan_us(c, p, T);
                if (t < us) us = t, best = p;
            }
    return best;
}

double enc_transforms_us(const CtxDev &c, size_t T) {
    const EncPlan p = enc_plan(c, T);
    return p.clusters ? enc_plan_us(c, p, T) : 0.0;
}

template <int CL>
static size_t ring_scratch(const CtxDev &c, size_t T) {
    using G = EncRing<CL>;
    size_t most = 0;                                   // of any number of ciphertexts up to T, on any plan
    for (uint32_t S = 1; S <= ENC_MOST; S++) {
        const uint32_t units = 2 * c.enc->way[c.enc->count - 1].units;
        if (S == 1 && enc_plan_by_size(c, T).S > 1) continue;
        const size_t want = T * ((units + S - 1) / S), fit = c.enc_fit[0][S], bytes = (want < fit ? want : fit) * (G::SHARED + S * G::OWN);
        if (bytes > most) most = bytes;
    }
    return most;
}
// ciphertexts whose samples are made ahead at once
constexpr size_t ENC_SAMPLE_BYTES = (size_t)256 << 20;
template <int CL>
static size_t ring_samples(size_t T) {
    const size_t most = ENC_SAMPLE_BYTES / EncRing<CL>::SAMPLES;
    return T < most ? T : most;
}
template <int CL>
static size_t ring_work(const CtxDev &c, size_t T) {
    const size_t a = ring_scratch<CL>(c, T) + ring_samples<CL>(T) * EncRing<CL>::SAMPLES, b = encrypt_passes_work_bytes(c, T);
    return a > b ? a : b;
}
size_t fft_work_bytes(const CtxDev &c, size_t T) {
    if (T == 0) return 0;
    FEDHE_FOR_RING(c, ring_work, c, T)
}

template <int CL>
static cudaError_t launch_encrypt_part(const CtxDev &c, const KeysDev &k, const float *sel, unsigned char *work, uint32_t t0,
                                       size_t T, uint64_t seed, uint32_t client, uint64_t *ct, cudaStream_t s) {
    using G = EncRing<CL>;
    static_assert(G::SAMPLES % 16 == 0, "scratch behind the samples, and e1 in 16-byte words");
    const EncPlan p = enc_plan(c, T);
    if (p.clusters < 1) return cudaErrorLaunchOutOfResources;
    cudaError_t e;
    // Few ciphertexts are drawn by their clusters: the launch costs the host more than the clusters take (N = 8192, a round of three
    // clients with 25 ciphertexts each: 170 us, and 193 us with three more launches).  With enough of them it pays: 100
    // ciphertexts of N = 8192 69.7 -> 63.5 us, 40 of N = 16384 72.7 -> 66.1, 68 of N = 32768 303 -> 267.
    EncDraw draw = {seed, client, t0, T * G::N < (size_t)1 << 19};
    if (!draw.inside) {
        const size_t items = T * G::ITEMS, fill = (size_t)c.sm_count * 8;
        enc_sample_kernel<CL><<<(unsigned)(items < fill ? items : fill), G::NT, 0, s>>>(c.gauss, draw, (uint32_t)T, work);
        if ((e = FEDHE_LAUNCHED())) return e;
    }
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute attr[2];
    cfg.stream = s;
    cfg.blockDim = dim3(G::NT, 1, 1);
    cfg.gridDim = dim3(p.clusters * p.S, 1, 1);
    cfg.dynamicSmemBytes = p.alone ? ENC_ALONE_SMEM : G::SMEM;
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = p.S;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    // The clusters start beside the last samples if there is one to a ciphertext.  With more, all the clusters that fit have to be there
    // at once, and those that come first may leave no room for a whole one (200 ciphertexts of N = 32768: 784 -> 800 us).
    cfg.numAttrs = !draw.inside && T <= p.clusters ? 2 : 1;
    if ((e = cudaLaunchKernelEx(&cfg, pairs_limbs(c, p.way) ? encrypt_fft_kernel<CL, true> : encrypt_fft_kernel<CL, false>, c, EncTable{c.enc_jobs + p.way,
                                c.enc->way[p.way].products}, k, sel, draw, work, work + T * G::SAMPLES, ct, (uint32_t)T, p.S, p.parts)))
        return e;
    return FEDHE_LAUNCHED();
}
template <int CL>
static cudaError_t launch_encrypt_ring(const CtxDev &c, const KeysDev &k, const float *sel, void *work, uint32_t t0,
                                       size_t T, uint64_t seed, uint32_t client, uint64_t *ct, cudaStream_t s) {
    using G = EncRing<CL>;
    const size_t most = ring_samples<CL>(T);
    for (size_t t = 0; t < T; t += most) {
        const cudaError_t e = launch_encrypt_part<CL>(c, k, sel + t * G::n, static_cast<unsigned char *>(work), t0 + (uint32_t)t,
                                                      T - t < most ? T - t : most, seed, client, ct + t * 2 * c.L * G::N, s);
        if (e) return e;
    }
    return cudaSuccess;
}

cudaError_t launch_encrypt(const CtxDev &c, const KeysDev &k, const float *sel, void *work, uint32_t t0, size_t T,
                           uint64_t seed, uint32_t client, uint64_t *ct, cudaStream_t s) {
    if (T == 0) return cudaSuccess;
    if (encrypt_by_passes(c, T)) return launch_encrypt_passes(c, k, sel, work, t0, T, seed, client, ct, s);
    FEDHE_FOR_RING(c, launch_encrypt_ring, c, k, sel, work, t0, T, seed, client, ct, s)
}

template <int CL>
static cudaError_t launch_decrypt_ring(const CtxDev &c, const KeysDev &k, const uint64_t *ct, uint32_t level, size_t T,
                                       double *z, cudaStream_t s) {
    using G = FftRing<CL>;
    auto kern = decrypt_fft_kernel<CL>;
    const size_t fit = c.enc_fit[0][G::R], clusters = T < fit ? T : fit;       // of the same shape as encryption's
    if (clusters < 1) return cudaErrorLaunchOutOfResources;
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute attr;
    cfg.stream = s;
    cfg.blockDim = dim3(G::NT, 1, 1);
    cfg.gridDim = dim3((unsigned)(clusters * G::R), 1, 1);
    cfg.dynamicSmemBytes = G::SMEM;
    attr.id = cudaLaunchAttributeClusterDimension;
    attr.val.clusterDim.x = G::R;
    attr.val.clusterDim.y = 1;
    attr.val.clusterDim.z = 1;
    cfg.attrs = &attr;
    cfg.numAttrs = G::R > 1 ? 1 : 0;
    cudaError_t e;
    if ((e = cudaLaunchKernelEx(&cfg, kern, c, k, ct, level, z, (uint32_t)T))) return e;
    return FEDHE_LAUNCHED();
}

// At N = 2^16 a ciphertext takes a cluster of eight blocks, the device holds 33 of them (15 with their SMs to themselves), and c1
// of 60 bits needs three pieces, so that the kernels of launch_decrypt(), which share out every ciphertext, are often faster.
// Measured (us, those and the transforms):
//   three pieces: 1, 14, 18, 28, 37, 75, 150, 600 ciphertexts   89 104, 99 98, 104 117, 139 117, 149 213, 296 320, 540 557, 1984 2055
//   two pieces: 1, 14, 28, 37, 56, 110, 300, 600                71 80, 83 74, 114 88, 122 143, 186 171, 298 313, 827 762, 1572 1452
// Both sides below are lines and steps through these.
bool decrypt_by_passes(const CtxDev &c, size_t T) {
    const uint32_t pieces = c.dec_split.pieces, fit = c.enc_fit[0][8], alone = c.enc_fit[1][8];
    if (c.logN < 16 || pieces < 2 || fit < 1) return false;
    const bool three = pieces > 2;
    const double t = (double)T, rounds = (double)((T + fit - 1) / fit);
    const double transforms = T <= alone ? (three ? 98.0 : 75.0) : T <= fit ? (three ? 118.0 : 90.0) : three ? 36.0 + 105.0 * rounds : 26.0 + 78.0 * rounds;
    const double passes = T <= 18 ? (three ? 88.0 : 70.0) + t : T <= 37 ? (three ? 105.0 + 1.25 * t : 85.0 + 1.07 * t) : three ? 45.0 + 3.3 * t : 47.0 + 2.6 * t;
    return passes < transforms;
}

cudaError_t launch_decrypt_fft(const CtxDev &c, const KeysDev &k, const uint64_t *ct, uint32_t level, size_t T,
                               double *z, cudaStream_t s) {
    if (T == 0) return cudaSuccess;
    FEDHE_FOR_RING(c, launch_decrypt_ring, c, k, ct, level, T, z, s)
}

__global__ void __launch_bounds__(256) gauss_table_kernel(GaussTables *g) { gauss_tables_init(*g, threadIdx.x, blockDim.x); }
size_t gauss_table_bytes() { return sizeof(GaussTables); }
cudaError_t launch_gauss_table(void *table, cudaStream_t s) {
    gauss_table_kernel<<<1, 256, 0, s>>>(static_cast<GaussTables *>(table));
    return FEDHE_LAUNCHED();
}

// ---- key tables ------------------------------------------------------------------------

// One thread block per (polynomial, block of its transform).  `pk`: the public key's coefficients
// [2][L][N], canonical; polynomial number -> (unit, component, product) in the order of the tables;
// the last one is the secret key.
template <int CL>
__global__ void __launch_bounds__(FftLay::NT)
fft_key_kernel(const __grid_constant__ CtxDev c, const __grid_constant__ EncWay way, const uint64_t *pk, const int8_t *s8, double2 *fft_pk, double2 *fft_s) {
    using G = FftRing<CL>;
    constexpr uint32_t NB = G::NB, NT = G::NT, R = G::R, n = G::n;
    extern __shared__ __align__(128) unsigned char smem[];
    double2 *buf = reinterpret_cast<double2 *>(smem);
    const uint32_t tid = threadIdx.x, b = blockIdx.x % R;
    uint32_t poly = blockIdx.x / R, u = 0;
    while (u < way.units && poly >= 2 * way.unit[u].products) poly -= 2 * way.unit[u++].products;
    const bool secret = u == way.units;
    const EncUnit &e = way.unit[secret ? 0 : u];
    const uint32_t comp = secret ? 0 : poly / e.products, product = secret ? 0 : poly % e.products;
    auto piece = [&](uint32_t second, uint32_t of, uint32_t i) {
        const uint32_t j = second ? e.limb2 : e.limb;
        const uint64_t v = pk[((size_t)comp * c.L + j) * c.N + i], q = c.limb[j].q;
        return fft_piece(c.limb[j].split[way.units < c.L], v > q / 2 ? (int64_t)(v - q) : (int64_t)v, of);
    };
    auto value = [&](uint32_t i) {
        if (secret) return (double)s8[i];
        if (e.limb2 == NO_LIMB) return (double)piece(0, product, i);
        if (product == 0) return (double)(piece(0, 0, i) + 65536 * piece(1, 0, i));
        return (double)piece(product == 1 ? 0 : 1, 1, i);
    };
    const OuterPath<CL> outer(c.fft_fwd, b);
    // the columns, in a loop, wait in the thread's own words of the buffer
#pragma unroll 1
    for (int r = 0; r < 16; r++) {
        cpx z[R];
#pragma unroll
        for (uint32_t a = 0; a < R; a++) {
            const uint32_t i = a * NB + tid + NT * r;
            z[a] = cpx{value(i), value(i + n)};
        }
        const cpx v = outer.apply(z);
        buf[tid + NT * r] = make_double2(v.re, v.im);
    }
    cpx x[16];
#pragma unroll
    for (int r = 0; r < 16; r++) x[r] = cpx{buf[tid + NT * r].x, buf[tid + NT * r].y};
    fft_forward<CL, true>(x, buf, c.fft_fwd, b, tid);
    double2 *dst = (secret ? fft_s : fft_pk + e.fft_key + (size_t)poly * n) + (size_t)b * NB + tid;
    const double scale = 1.0 / n;                  // a power of two
#pragma unroll
    for (int r = 0; r < 16; r++) dst[r * NT] = make_double2(x[r].re * scale, x[r].im * scale);
}

template <int CL>
static cudaError_t launch_fft_keys_ring(const CtxDev &c, const uint64_t *pk, const int8_t *s8, double2 *fft_pk,
                                        double2 *fft_s, cudaStream_t s) {
    using G = FftRing<CL>;
    const size_t smem = (size_t)G::NB * 16;
    cudaError_t e;
    if ((e = cudaFuncSetAttribute(fft_key_kernel<CL>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem))) return e;
    for (uint32_t i = 0; i < c.enc->count; i++) {         // the secret with the first
        const EncWay &way = c.enc->way[i];
        fft_key_kernel<CL><<<(2 * way.products + (i == 0 ? 1 : 0)) * G::R, G::NT, smem, s>>>(c, way, pk, s8, fft_pk, fft_s);
        if ((e = FEDHE_LAUNCHED())) return e;
    }
    return cudaSuccess;
}

cudaError_t launch_fft_keys(const CtxDev &c, const uint64_t *pk, const int8_t *s8, double2 *fft_pk, double2 *fft_s,
                            cudaStream_t s) {
    FEDHE_FOR_RING(c, launch_fft_keys_ring, c, pk, s8, fft_pk, fft_s, s)
}

}  // namespace fedhe

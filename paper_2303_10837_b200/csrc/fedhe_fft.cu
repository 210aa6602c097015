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

__device__ __forceinline__ cpx fft_mul(double2 a, double2 b) { return cpx_mul(cpx{a.x, a.y}, b.x, b.y); }

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
    __device__ __forceinline__ FftJoin(const FftSplit &f, uint64_t q) : minus_q(0 - q), scale(f.top_scale), shift(f.shift[f.pieces - 1]) {
        // the quotient carries 2^17, which keeps it positive
        fix = (q << 17) - ((uint64_t)FFT_ROUND_BITS << shift);
    }
    __device__ __forceinline__ int64_t operator()(int64_t v, double z) const {
        const uint32_t k = (uint32_t)__double_as_longlong(f64_fma(z, scale, FFT_ROUND + 131072.0));
        return (int64_t)((uint64_t)v + fix + ((uint64_t)fft_round_bits(z) << shift) + (uint64_t)k * minus_q);
    }
};

// the residue in [0, q) of |v| < q
__device__ __forceinline__ uint64_t fft_canonical(int64_t v, uint64_t q) { return (uint64_t)(v + ((v >> 63) & (int64_t)q)); }

// geometry of a ring: a cluster of R thread blocks, one per block of the transform
template <int CL_>
struct FftRing {
    using Tab = FftTab<CL_>;
    static constexpr int CL = CL_, R = 1 << CL, NB = FftLay::NB, NT = FftLay::NT, n = R * NB, N = 2 * n;
    static constexpr int PER = 16 / R, COLS = NB / R;     // columns of the R x NB view that a thread, a thread block finishes
    // scratch in global memory (it lives in L2): a thread block's, then a cluster's
    static constexpr size_t UHAT = (size_t)NB * 16, PARK = (size_t)NB * 16, OWN = UHAT + PARK, TERMS = (size_t)N * 8,
                            UBITS = (size_t)NB * 4, SCRATCH = R * OWN + TERMS + UBITS;
    static constexpr size_t SMEM = (size_t)NB * 16 + (size_t)Tab::WORDS * 16;
    static constexpr int BATCH = 8;                       // coefficients whose loads are in flight together
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
// the same in the block's own order of the coefficients it finishes: [2 halves][R rows][COLS]
template <class G>
__device__ __forceinline__ uint32_t fft_own(int i) {
    const int o = i >> 1;
    return (o % G::R) * G::COLS + G::NT * (o / G::R) + (i & 1) * G::NB;
}

// ---- joined lower pieces, parked for the thread that will join the top one ----
template <class G>
__device__ __forceinline__ void fft_park(const cpx (&x)[16], unsigned char *park, const FftSplit &f, uint32_t piece,
                                         uint32_t tid) {
    if (f.narrow) {
        int *p = reinterpret_cast<int *>(park) + tid;
#pragma unroll
        for (int i = 0; i < 32; i++) __stcg(p + i * G::NT, (int)fft_round_bits((i & 1) ? x[i >> 1].im : x[i >> 1].re));
    } else {
        long long *p = reinterpret_cast<long long *>(park) + tid;
        const uint32_t sh = f.shift[piece];
#pragma unroll
        for (int i = 0; i < 32; i++) {
            long long w = (fft_round_bits((i & 1) ? x[i >> 1].im : x[i >> 1].re) - FFT_ROUND_BITS) << sh;
            if (piece) w += __ldcg(p + i * G::NT);
            __stcg(p + i * G::NT, w);
        }
    }
}
// val += the parked sums of values i0 .. i0 + BATCH - 1
template <class G>
__device__ __forceinline__ void fft_parked(int64_t (&val)[G::BATCH], const unsigned char *park, const FftSplit &f, int i0,
                                           uint32_t tid) {
    if (f.narrow) {
#pragma unroll
        for (int i = 0; i < G::BATCH; i++) val[i] += __ldcg(reinterpret_cast<const int *>(park) + (i0 + i) * G::NT + tid);
    } else if (f.pieces > 1) {
#pragma unroll
        for (int i = 0; i < G::BATCH; i++) val[i] += __ldcg(reinterpret_cast<const long long *>(park) + (i0 + i) * G::NT + tid);
    }
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

// The work of an encryption is dealt out in units (ciphertext, component, limb), weighed by their pieces:
// first unit that begins at or after `pos` pieces of [ciphertext][component][limb][piece].
__device__ __forceinline__ uint32_t fft_unit_at(const CtxDev &c, uint64_t pos) {
    const uint32_t half = c.fft_pieces;
    const uint32_t hc = (uint32_t)(pos / half);               // (ciphertext, component)
    uint32_t rest = (uint32_t)(pos % half), j = 0;
    while (rest) {
        const uint32_t p = c.limb[j].split.pieces;
        rest = rest > p ? rest - p : 0;
        j++;
    }
    return hc * c.L + j;
}

// A cluster of R thread blocks owns a range of (ciphertext, component, limb) units.  Per ciphertext: u is
// drawn and transformed once (its transform waits in the blocks' scratch, i.e. in L2, read back by the threads
// that wrote it), the slots are encoded in the transform buffers; per component the error terms are drawn,
// e0 added to the message; per unit and piece of the key: product with the key's table, inverse transform,
// rounding, joining, error and message terms, canonical residue.  HBM sees the slots and the ciphertext
// once.  A cluster whose range begins inside a ciphertext repeats what it needs of the ciphertext's preparation.
//
// Two thread blocks fit on an SM on every ring, so that one's memory phases meet the other's arithmetic, and
// what all of them keep in scratch (54 MB) stays in L2.
template <int CL>
__global__ void __launch_bounds__(FftLay::NT, 2)
encrypt_fft_kernel(const __grid_constant__ CtxDev c, const KeysDev k, const float *sel, unsigned char *work,
                   uint32_t t0, uint64_t seed, uint32_t client, uint64_t *ct, uint32_t T) {
    using G = FftRing<CL>;
    constexpr uint32_t N = G::N, n = G::n, NB = G::NB, NT = G::NT, R = G::R;
    extern __shared__ __align__(128) unsigned char smem[];
    double2 *buf = reinterpret_cast<double2 *>(smem);
    root_t *tab = reinterpret_cast<root_t *>(smem + (size_t)NB * 16);
    __shared__ GaussTables gt;
    __shared__ __align__(16) int8_t samples[2 * G::NB];   // e1 of the coefficients this block finishes
    const uint32_t rank = blockIdx.x % R, cid = blockIdx.x / R, nc = gridDim.x / R;
    gauss_tables_init(gt, threadIdx.x, NT);
    for (uint32_t i = threadIdx.x; i < (uint32_t)G::Tab::WORDS; i += NT) tab[i] = c.fft_inv[i];
    buffer_free<CL>();
    unsigned char *shared_work = work + (size_t)cid * G::SCRATCH, *own = shared_work + rank * G::OWN;
    double2 *uhat = reinterpret_cast<double2 *>(own);                           // [16][NT]
    unsigned char *park = own + G::UHAT;
    // message and e0 by residue of the coefficient's number: [2 halves][R][NB], coefficient R kk + b at kk of row b
    long long *terms = reinterpret_cast<long long *>(shared_work + R * G::OWN);
    // u, two bits (value + 1) per row of the column: [2 halves][NB]
    uint16_t *ubits = reinterpret_cast<uint16_t *>(shared_work + R * G::OWN + G::TERMS);
    auto term_of = [&](uint32_t coef) {
        return terms + ((coef & (n - 1)) >> CL) + ((coef & (R - 1)) + (coef >= n ? R : 0)) * NB;
    };

    const uint32_t per_ct = 2 * c.L;
    const uint64_t total = (uint64_t)T * 2 * c.fft_pieces;
    const uint32_t u_end = fft_unit_at(c, total * (cid + 1) / nc);
    uint32_t have_ct = 0xffffffffu, have_e = 0xffffffffu;
    bool big = false;                                     // a term of this component needs reducing first
#pragma unroll 1
    for (uint32_t unit = fft_unit_at(c, total * cid / nc); unit < u_end; unit++) {
        const uint32_t tl = unit / per_ct, comp = (unit / c.L) & 1u, j = unit % c.L, t = t0 + tl;
        if (tl != have_ct) {
            have_ct = tl;
            // four columns of one half at a time
#pragma unroll 1
            for (uint32_t w = rank * (2 * NB / 4 / R) + threadIdx.x; w < (rank + 1) * (2 * NB / 4 / R); w += NT) {
                uint32_t f[4] = {0, 0, 0, 0};
#pragma unroll
                for (uint32_t a = 0; a < R; a++) {
                    const uint32_t b = (w / (NB / 4)) * (n / 4) + a * (NB / 4) + w % (NB / 4);
                    const u32x4 v = stream_block(seed, b, t, client, TAG_ENC_U);
                    f[0] |= (uint32_t)(ternary_from_word(v.x) + 1) << (2 * a);
                    f[1] |= (uint32_t)(ternary_from_word(v.y) + 1) << (2 * a);
                    f[2] |= (uint32_t)(ternary_from_word(v.z) + 1) << (2 * a);
                    f[3] |= (uint32_t)(ternary_from_word(v.w) + 1) << (2 * a);
                }
                __stcg(reinterpret_cast<uint2 *>(ubits) + w, make_uint2(f[0] | f[1] << 16, f[2] | f[3] << 16));
            }
            cluster_meet<CL>();                           // u is there, and nobody reads the last ciphertext's terms any more
            cpx x[16];
            {
                const OuterPath<CL> outer(c.fft_fwd, rank);
                const uint16_t *p = ubits + fresh_tid();
                auto ternary = [](uint32_t f) {           // 0, 1, 2 -> -1.0, 0.0, 1.0
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
            fft_forward<CL>(x, buf, c.fft_fwd, rank, fresh_tid());
            {
                double2 *dst = uhat + fresh_tid();
#pragma unroll
                for (int r = 0; r < 16; r++) __stcg(dst + r * NT, make_double2(x[r].re, x[r].im));
            }
            if (comp == 0) {
                const float *slots = sel + (size_t)tl * n;
                long long *row = terms + (CL ? bitrev(rank, CL ? CL : 1) : 0u) * NB;
                buffer_wait<CL>();
                if (encode_block_in_place<Lay<FftLay::LB, 4>>(
                        c, [&](uint32_t i) { return encoder_stages<CL>(slots, c.ftw, n, rank, i); },
                        reinterpret_cast<uint64_t *>(buf), CL,
                        [&](uint32_t kk, int64_t re, int64_t im) {
                            __stcg(row + kk, (long long)re);
                            __stcg(row + R * NB + kk, (long long)im);
                        }))
                    atomicOr(c.status, 1);
                buffer_free<CL>();
                if constexpr (CL > 0) cluster_meet<CL>(); // the message of all blocks is complete
            }
        }
        if (2 * tl + comp != have_e) {
            have_e = 2 * tl + comp;
            __syncthreads();                              // nobody still reads the samples
            int far = 0;
            // pairs of neighbours among the coefficients this block finishes: [2 R rows][COLS]
            for (uint32_t pp = threadIdx.x; pp < NB; pp += NT) {
                const uint32_t row = pp / (G::COLS / 2), lc = 2 * (pp % (G::COLS / 2));
                const uint32_t coef = row * NB + rank * G::COLS + lc;
                const u32x4 w = stream_block(seed, coef >> 1, t, client, comp == 0 ? TAG_ENC_E0 : TAG_ENC_E1);
                const int ex = gauss_from_u64(gt, (uint64_t)w.x | ((uint64_t)w.y << 32));
                const int ey = gauss_from_u64(gt, (uint64_t)w.z | ((uint64_t)w.w << 32));
                if (comp == 0) {
                    long long *px = term_of(coef), *py = term_of(coef + 1);
                    const long long mx = __ldcg(px) + ex, my = __ldcg(py) + ey;
                    far |= (mx < 0 ? -mx : mx) >= c.term_limit || (my < 0 ? -my : my) >= c.term_limit;
                    __stcg(px, mx);
                    __stcg(py, my);
                } else {
                    *reinterpret_cast<char2 *>(samples + row * G::COLS + lc) = make_char2((signed char)ex, (signed char)ey);
                }
            }
            big = __syncthreads_or(far);                  // and the samples and terms are complete
        }
        const FftSplit &f = c.limb[j].split;
        const uint64_t q = c.limb[j].q;
#pragma unroll 1
        for (uint32_t p = 0; p < f.pieces; p++) {
            cpx x[16];
            {
                const uint32_t tid = fresh_tid();
                const double2 *key = k.fft_pk + c.limb[j].fft_key + ((size_t)(comp * f.pieces + p) * R + rank) * NB + tid;
                const double2 *uh = uhat + tid;
#pragma unroll
                for (int r = 0; r < 16; r++) x[r] = fft_mul(__ldcg(uh + r * NT), load_passing(key + r * NT));
            }
            fft_inverse<CL>(x, buf, tab, fresh_tid());
            const uint32_t tid = fresh_tid();
            fft_gather<G>(x, buf, tab, rank, tid);
            if (p + 1 < f.pieces) {
                fft_park<G>(x, park, f, p, tid);
                continue;
            }
            uint64_t *out = ct + (((size_t)tl * 2 + comp) * c.L + j) * N + tid;
            const FftJoin join(f, q);
#pragma unroll
            for (int i0 = 0; i0 < 32; i0 += G::BATCH) {
                int64_t val[G::BATCH];
                if (comp == 1) {
#pragma unroll
                    for (int i = 0; i < G::BATCH; i++) val[i] = samples[fft_own<G>(i0 + i) + tid];
                } else if (big) {
#pragma unroll
                    for (int i = 0; i < G::BATCH; i++) val[i] = 0;
                } else {
#pragma unroll
                    for (int i = 0; i < G::BATCH; i++) val[i] = __ldcg(term_of(fft_coefficient<G>(i0 + i, rank) + tid));
                }
                fft_parked<G>(val, park, f, i0, tid);
                // streaming stores: the finished ciphertext should not push tables and scratch out of L2
#pragma unroll
                for (int i = 0; i < G::BATCH; i++) {
                    const cpx &w = x[(i0 + i) >> 1];
                    val[i] = join(val[i], (i & 1) ? w.im : w.re);
                    __stcs(reinterpret_cast<unsigned long long *>(out + fft_coefficient<G>(i0 + i, rank)),
                           (unsigned long long)fft_canonical(val[i], q));
                }
            }
            if (big && comp == 0) {
                // terms beyond a quarter of the smallest prime: encoded updates are far below, so this is rare
                const uint64_t mu = c.limb[j].mu;
#pragma unroll 1
                for (int i = 0; i < 32; i++) {
                    const uint32_t at = fft_coefficient<G>(i, rank);
                    out[at] = addmod(out[at], signed_residue(__ldcg(term_of(at + tid)), q, mu), q);
                }
            }
        }
    }
    buffer_wait<CL>();                                    // the other blocks have read this one's buffer
}

// ===========================================================================
// decryption + decoding:  d = c0 + c1 s on limb 0, centred, then the slot transform
// ===========================================================================

// A cluster decrypts and decodes a range of ciphertexts: per piece of c1 a forward
// transform, the product with the transformed secret, an inverse transform; joining, c0, centring;
// then the slot transform, which is the forward transform again (a slot is the value at one of the
// roots; `slot_of` puts the values in order through shared memory).  Only the two limb-0
// polynomials are read and the n decoded values written.
template <int CL>
__global__ void __launch_bounds__(FftLay::NT, 2)
decrypt_fft_kernel(const __grid_constant__ CtxDev c, const KeysDev k, const uint64_t *ct, uint32_t level,
                   unsigned char *work, double *z, uint32_t T) {
    using G = FftRing<CL>;
    constexpr uint32_t n = G::n, NB = G::NB, NT = G::NT, R = G::R;
    constexpr size_t N = G::N;
    extern __shared__ __align__(128) unsigned char smem[];
    double2 *buf = reinterpret_cast<double2 *>(smem);
    root_t *tab = reinterpret_cast<root_t *>(smem + (size_t)NB * 16);
    const uint32_t rank = blockIdx.x % R, cid = blockIdx.x / R, nc = gridDim.x / R;
    for (uint32_t i = threadIdx.x; i < (uint32_t)G::Tab::WORDS; i += NT) tab[i] = c.fft_inv[i];
    buffer_free<CL>();
    unsigned char *park = work + (size_t)cid * G::SCRATCH + rank * G::OWN + G::UHAT;
    const FftSplit &f = c.dec_split;
    const uint64_t q = c.limb[0].q;
    const int64_t half_q = (int64_t)(q / 2);
    const double inv_delta = __longlong_as_double((long long)(1023 - c.log2_delta) << 52);
    const uint32_t t_end = (uint32_t)((uint64_t)T * (cid + 1) / nc);
    __syncthreads();
#pragma unroll 1
    for (uint32_t t = (uint32_t)((uint64_t)T * cid / nc); t < t_end; t++) {
        const uint64_t *c0 = ct + ((size_t)t * 2 * level) * N, *c1 = c0 + level * N;
        cpx x[16];
        // the pieces, then the slot transform as one more turn of the same code
#pragma unroll 1
        for (uint32_t p = 0; p <= f.pieces; p++) {
            if (p < f.pieces) {
                const uint64_t *src = c1 + fresh_tid();
                auto value = [&](uint64_t v) {
                    return fft_from_int(fft_piece(f, v > (uint64_t)half_q ? (int64_t)(v - q) : (int64_t)v, p));
                };
#pragma unroll
                for (int o = 0; o < 16; o++) {
                    const uint64_t re = __ldg(src + fft_coefficient<G>(2 * o, rank)), im = __ldg(src + fft_coefficient<G>(2 * o + 1, rank));
                    x[o] = cpx{value(re), value(im)};
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
            const uint32_t tid = fresh_tid();
            fft_gather<G>(x, buf, tab, rank, tid);
            if (p + 1 < f.pieces) {
                fft_park<G>(x, park, f, p, tid);
                continue;
            }
            const FftJoin join(f, q);
#pragma unroll
            for (int i0 = 0; i0 < 32; i0 += G::BATCH) {
                int64_t val[G::BATCH];
#pragma unroll
                for (int i = 0; i < G::BATCH; i++) val[i] = (int64_t)__ldg(c0 + fft_coefficient<G>(i0 + i, rank) + tid);
                fft_parked<G>(val, park, f, i0, tid);
#pragma unroll
                for (int i = 0; i < G::BATCH; i++) {
                    cpx &w = x[(i0 + i) >> 1];
                    int64_t d = join(val[i], (i & 1) ? w.im : w.re);      // (-q, 2q)
                    d -= d > half_q ? (int64_t)q : 0;
                    d -= d > half_q ? (int64_t)q : 0;
                    d += d < -half_q ? (int64_t)q : 0;
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
}

// ---- launch --------------------------------------------------------------------------

#define FEDHE_FOR_RING(c, FN, ...)                          \
    switch ((c).logN) {                                     \
    case 13: return FN<0>(__VA_ARGS__);                     \
    case 14: return FN<1>(__VA_ARGS__);                     \
    case 15: return FN<2>(__VA_ARGS__);                     \
    default: return FN<3>(__VA_ARGS__);                     \
    }

// as many clusters as the device holds at once, no more than there is work
template <class G, class K>
static cudaError_t fft_grid(K kern, int n_sm, size_t want, cudaStream_t s, cudaLaunchConfig_t &cfg, cudaLaunchAttribute *attr) {
    cudaError_t e;
    if ((e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)G::SMEM))) return e;
    cfg = {};
    cfg.stream = s;
    cfg.blockDim = dim3(G::NT, 1, 1);
    cfg.dynamicSmemBytes = G::SMEM;
    size_t fit = 2 * (size_t)n_sm / G::R;
    if constexpr (G::CL > 0) {
        attr->id = cudaLaunchAttributeClusterDimension;
        attr->val.clusterDim.x = G::R;
        attr->val.clusterDim.y = 1;
        attr->val.clusterDim.z = 1;
        cfg.attrs = attr;
        cfg.numAttrs = 1;
        if (want > fit / 2) {
            cfg.gridDim = dim3(G::R, 1, 1);
            int clusters = 0;
            if ((e = cudaOccupancyMaxActiveClusters(&clusters, kern, &cfg))) return e;
            if (clusters < 1) return cudaErrorLaunchOutOfResources;
            if ((size_t)clusters < fit) fit = (size_t)clusters;
        }
    }
    cfg.gridDim = dim3((unsigned)((want < fit ? want : fit) * G::R), 1, 1);
    return cudaSuccess;
}

template <int CL>
static size_t ring_scratch(int n_sm, size_t units) {
    const size_t fit = 2 * (size_t)n_sm / FftRing<CL>::R;
    return (units < fit ? units : fit) * FftRing<CL>::SCRATCH;
}
size_t fft_work_bytes(const CtxDev &c, int n_sm, size_t T) { FEDHE_FOR_RING(c, ring_scratch, n_sm, T * 2 * c.L) }

template <int CL>
static cudaError_t launch_encrypt_ring(const CtxDev &c, const KeysDev &k, const float *sel, void *work, int n_sm, uint32_t t0,
                                       size_t T, uint64_t seed, uint32_t client, uint64_t *ct, cudaStream_t s) {
    auto kern = encrypt_fft_kernel<CL>;
    cudaLaunchConfig_t cfg;
    cudaLaunchAttribute attr;
    cudaError_t e;
    if ((e = fft_grid<FftRing<CL>>(kern, n_sm, T * 2 * c.L, s, cfg, &attr))) return e;
    if ((e = cudaLaunchKernelEx(&cfg, kern, c, k, sel, static_cast<unsigned char *>(work), t0, seed, client, ct, (uint32_t)T)))
        return e;
    return FEDHE_LAUNCHED();
}

cudaError_t launch_encrypt(const CtxDev &c, const KeysDev &k, const float *sel, void *work, int n_sm,
                           uint32_t t0, size_t T, uint64_t seed, uint32_t client, uint64_t *ct,
                           cudaStream_t s) {
    if (T == 0) return cudaSuccess;
    FEDHE_FOR_RING(c, launch_encrypt_ring, c, k, sel, work, n_sm, t0, T, seed, client, ct, s)
}

template <int CL>
static cudaError_t launch_decrypt_ring(const CtxDev &c, const KeysDev &k, const uint64_t *ct, uint32_t level, size_t T,
                                       void *work, int n_sm, double *z, cudaStream_t s) {
    auto kern = decrypt_fft_kernel<CL>;
    cudaLaunchConfig_t cfg;
    cudaLaunchAttribute attr;
    cudaError_t e;
    if ((e = fft_grid<FftRing<CL>>(kern, n_sm, T, s, cfg, &attr))) return e;
    if ((e = cudaLaunchKernelEx(&cfg, kern, c, k, ct, level, static_cast<unsigned char *>(work), z, (uint32_t)T))) return e;
    return FEDHE_LAUNCHED();
}

cudaError_t launch_decrypt_fft(const CtxDev &c, const KeysDev &k, const uint64_t *ct, uint32_t level, size_t T,
                               void *work, int n_sm, double *z, cudaStream_t s) {
    if (T == 0) return cudaSuccess;
    FEDHE_FOR_RING(c, launch_decrypt_ring, c, k, ct, level, T, work, n_sm, z, s)
}

// ---- key tables ------------------------------------------------------------------------

// One thread block per (polynomial, block of its transform).  `pk`: the public key's coefficients
// [2][L][N], canonical; polynomial number -> (limb, component, piece) in the order of the tables;
// the last one is the secret key.
template <int CL>
__global__ void __launch_bounds__(FftLay::NT)
fft_key_kernel(const __grid_constant__ CtxDev c, const uint64_t *pk, const int8_t *s8, double2 *fft_pk, double2 *fft_s) {
    using G = FftRing<CL>;
    constexpr uint32_t NB = G::NB, NT = G::NT, R = G::R, n = G::n;
    extern __shared__ __align__(128) unsigned char smem[];
    double2 *buf = reinterpret_cast<double2 *>(smem);
    const uint32_t tid = threadIdx.x, b = blockIdx.x % R;
    uint32_t poly = blockIdx.x / R, j = 0;
    while (j < c.L && poly >= 2 * c.limb[j].split.pieces) poly -= 2 * c.limb[j++].split.pieces;
    const bool secret = j == c.L;
    const LimbDev &lb = c.limb[secret ? 0 : j];
    const uint32_t comp = secret ? 0 : poly / lb.split.pieces, piece = secret ? 0 : poly % lb.split.pieces;
    const uint64_t *src = pk + ((size_t)comp * c.L + (secret ? 0 : j)) * c.N;
    auto value = [&](uint32_t i) {
        if (secret) return (double)s8[i];
        const uint64_t v = src[i];
        return (double)fft_piece(lb.split, v > lb.q / 2 ? (int64_t)(v - lb.q) : (int64_t)v, piece);
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
    double2 *dst = (secret ? fft_s : fft_pk + lb.fft_key + (size_t)poly * n) + (size_t)b * NB + tid;
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
    fft_key_kernel<CL><<<(2 * c.fft_pieces + 1) * G::R, G::NT, smem, s>>>(c, pk, s8, fft_pk, fft_s);
    return FEDHE_LAUNCHED();
}

cudaError_t launch_fft_keys(const CtxDev &c, const uint64_t *pk, const int8_t *s8, double2 *fft_pk, double2 *fft_s,
                            cudaStream_t s) {
    FEDHE_FOR_RING(c, launch_fft_keys_ring, c, pk, s8, fft_pk, fft_s, s)
}

}  // namespace fedhe

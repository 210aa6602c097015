// Encryption into the transform-domain wire format, and into the coefficient format by passes where that is
// faster (part 3 of the kernels); the coefficient format otherwise is in fedhe_fft.cu.
#include "fedhe_kernels.cuh"
#include "fedhe_slots.cuh"

namespace fedhe {

// ===========================================================================
// encryption:  c0 = pk0 u + e0 + m,  c1 = pk1 u + e1   (mod every q_j), every limb transformed
// ===========================================================================

// Index swizzle of the one-byte sample arrays in shared memory (banks of four
// bytes, i.e. index bits 2..6): the first phase of a transform reads them with
// lanes that differ in index bits 0, 1, 7, 8 and 9, the epilogues with
// consecutive lanes; folding bits 7..9 into bits 2..4 keeps both patterns free
// of bank conflicts, leaves aligned groups of four intact, and does not involve
// the first phase's register bits (10 and up), so a thread computes it once.
__device__ __forceinline__ uint32_t bswz(uint32_t i) { return i ^ (((i >> 7) & 7u) << 2); }

// One (ciphertext, limb) unit in the limb's arithmetic, transform-domain output:
// c0^ = pk0^ u^ + (e0 + m)^, c1^ = pk1^ u^ + e1^.  Three passes over one copy of the
// forward-transform code: u (both products wait in their final slots), then e0 + m and
// e1, each added to its product.
template <class M, class L, int V>
__device__ __forceinline__ void encrypt_unit(const LimbDev &lb, const tw_t *p0, const tw_t *p1, uint64_t *sm,
                                             const int8_t *su, const int8_t *se0, const int64_t *mt,
                                             uint64_t *cbase, size_t cstride) {
    using val = typename M::val;
    constexpr uint32_t B = 1u << L::LOGB;
    const uint32_t tid = threadIdx.x;
    const uint64_t q = lb.q;
    const auto fa = LimbOf<M>::args(lb, true, 0, 0);
    const M &ar = fa.m;
#pragma unroll 1
    for (int h = 0; h < 3; h++) {
        uint64_t *cc = cbase + (h == 2 ? cstride : 0);
        const int8_t *se = se0 + (h == 2 ? B : 0);
        smem_ntt_forward<L, V>(
            sm, tid, fa,
            [&](uint32_t i) {
                if (h == 0) return ar.small(su[bswz(i)]);
                if (h == 2) return ar.small(se[bswz(i)]);
                return ar.from_residue(signed_residue(__ldcg(mt + i) + (int64_t)se[bswz(i)], q, lb.mu));
            },
            [&](uint32_t p, val a, val b) {
                if (h == 0) {
                    const auto a0 = M::load_key(p0 + p), a1 = M::load_key(p0 + p + 1);
                    const auto b0 = M::load_key(p1 + p), b1 = M::load_key(p1 + p + 1);
                    *reinterpret_cast<u64x2 *>(cbase + p) =
                        u64x2{M::bits(ar.mul_key(a, a0)), M::bits(ar.mul_key(b, a1))};
                    *reinterpret_cast<u64x2 *>(cbase + cstride + p) =
                        u64x2{M::bits(ar.mul_key(a, b0)), M::bits(ar.mul_key(b, b1))};
                } else {
                    const u64x2 t = *reinterpret_cast<const u64x2 *>(cc + p);
                    *reinterpret_cast<u64x2 *>(cc + p) =
                        u64x2{ar.canon_sum(a, M::from_bits(t.x)), ar.canon_sum(b, M::from_bits(t.y))};
                }
            });
        __syncthreads();   // last-phase readers are done before the next transform writes
    }
}

// Fused path for N <= 2^14 (one block holds a whole limb): a thread block
// draws u, e0, e1 of a ciphertext once into shared memory and encodes the
// ciphertext's slots (the slot transform runs in the limb buffer; the rounded
// message goes to a scratch of N words that belongs to this block alone and is
// read back once per limb, so it lives in L2), then does the three transforms of
// every limb of it.  A block whose range of units begins in the middle of a
// ciphertext encodes that ciphertext again for itself (no block waits for another).
template <class L, int V>
__global__ void __launch_bounds__(L::NT / V, (L::NT / V) <= 512 ? 2 : 1)
encrypt_fused_kernel(const __grid_constant__ CtxDev c, const KeysDev k, const float *sel, int64_t *mscr,
                     uint32_t t0, uint64_t seed, uint32_t client, uint64_t *ct, uint32_t T) {
    using LF = Lay<L::LOGB - 1, 3>;                  // the slot transform of the same ring
    static_assert(LF::NT == L::NT / V, "the encoder is played by the same threads");
    extern __shared__ __align__(128) uint64_t sm[];
    constexpr uint32_t B = 1u << L::LOGB, RT = L::NT / V;
    int8_t *su = reinterpret_cast<int8_t *>(sm + B);
    int8_t *se0 = su + B, *se1 = se0 + B;
    const uint32_t tid = threadIdx.x;
    __shared__ GaussTables gt;
    gauss_tables_load(gt, c.gauss, tid, blockDim.x);

    // Work units are (ciphertext, limb) pairs in ciphertext-major order, dealt
    // evenly to the blocks of the grid (one block per SM), so that the last
    // wave is as full as the others; a block re-draws u, e0, e1 whenever its
    // range moves on to the next ciphertext.
    const uint64_t units = (uint64_t)T * c.L;
    const uint32_t u_begin = (uint32_t)(units * blockIdx.x / gridDim.x);
    const uint32_t u_end = (uint32_t)(units * (blockIdx.x + 1) / gridDim.x);
    const size_t cstride = (size_t)c.L * B;          // from c0 to c1 of the same limb
    int64_t *mblk = mscr + (size_t)blockIdx.x * B;   // this block's encoded message (stays in L2)
    uint32_t sampled = 0xffffffffu;
    for (uint32_t unit = u_begin; unit < u_end; unit++) {
        const uint32_t tl = unit / c.L, j = unit % c.L;   // ciphertext within this call, limb
        if (tl != sampled) {
            sampled = tl;
            const uint32_t t = t0 + tl;                   // stream coordinate
            __syncthreads();                              // tables ready / previous samples no longer read
            for (uint32_t b = tid; b < B / 4; b += RT) {
                u32x4 w = stream_block(seed, b, t, client, TAG_ENC_U);
                char4 v = make_char4((signed char)ternary_from_word(w.x), (signed char)ternary_from_word(w.y),
                                     (signed char)ternary_from_word(w.z), (signed char)ternary_from_word(w.w));
                *reinterpret_cast<char4 *>(su + bswz(4 * b)) = v;
            }
            for (uint32_t b = tid; b < B / 2; b += RT) {
                const int2 a = gauss_pair(gt, seed, b, t, client, TAG_ENC_E0), e = gauss_pair(gt, seed, b, t, client, TAG_ENC_E1);
                *reinterpret_cast<char2 *>(se0 + bswz(2 * b)) = make_char2((signed char)a.x, (signed char)a.y);
                *reinterpret_cast<char2 *>(se1 + bswz(2 * b)) = make_char2((signed char)e.x, (signed char)e.y);
            }
            // the ciphertext's message: slot transform, scaling and rounding in the limb buffer
            if (encode_in_block<LF>(c, sel + (size_t)tl * (B / 2), sm, mblk)) atomicOr(c.status, STATUS_RANGE);
        }
        const LimbDev &lb = c.limb[j];
        uint64_t *cbase = ct + (((size_t)tl * 2 + 0) * c.L + j) * B;
        FEDHE_FOR_ARITH_SEL(lb, (encrypt_unit<M_, L, V>(lb, k.pk0_hat + (size_t)j * B, k.pk1_hat + (size_t)j * B, sm, su,
                                                    se0, mblk, cbase, cstride)));
    }
}

// One (ciphertext, limb) unit of the two-group kernel below (N = 2 * 2^LOGB).
template <class M, class L, int V>
__device__ __forceinline__ void encrypt_unit2(const LimbDev &lb, const tw_t *pk0, const tw_t *pk1, uint64_t *sm,
                                              const int8_t *su, const int8_t *se0, const int64_t *mt,
                                              uint64_t *cbase, size_t cstride) {
    using val = typename M::val;
    constexpr uint32_t H = 1u << L::LOGB, B = 2 * H;
    constexpr uint32_t GT = L::NT / V;
    const uint32_t tid = threadIdx.x;
    const uint32_t grp = tid / GT, gt = tid % GT;
    uint64_t *smg = sm + grp * H;                          // this group's half
    const GroupSync gsync = {1 + grp, GT};
    const uint64_t q = lb.q;
    const tw_t *p0 = pk0 + grp * H, *p1 = pk1 + grp * H;
    uint64_t *c0 = cbase + grp * H, *c1 = cbase + cstride + grp * H;
    const auto fa = LimbOf<M>::args(lb, true, 1, grp);
    const M &ar = fa.m;
    const auto w0 = M::load(fa.tw + 1);                    // twiddle of the stage that pairs the halves
#pragma unroll 1
    for (int h = 0; h < 3; h++) {
        uint64_t *cc = h == 2 ? c1 : c0;
        const int8_t *se = se0 + (h == 2 ? B : 0);
        auto value = [&](uint32_t i) {
            if (h == 2) return ar.small(se[bswz(i)]);
            return ar.from_residue(signed_residue(__ldcg(mt + i) + (int64_t)se[bswz(i)], q, lb.mu));
        };
        smem_ntt_forward<L, V>(
            smg, gt, fa,
            [&](uint32_t i) {
                if (h == 0) {
                    // u is ternary: the twiddle product is 0, w or -w
                    const int a = su[bswz(i)], b = su[bswz(i + H)];
                    if constexpr (std::is_same<M, ModF64>::value) {
                        return f64_fma(grp == 0 ? (double)b : (double)-b, w0, (double)a);
                    } else {
                        const uint64_t u = small_residue(a, q);
                        const uint64_t v = b == 0 ? 0 : (b > 0 ? w0.w : q - w0.w);
                        return grp == 0 ? u + v : u - v + ar.q2;
                    }
                }
                const val lo = value(i), hi = value(i + H);    // the pairing stage costs one product per element
                if constexpr (std::is_same<M, ModF64>::value) {
                    const double t = ar.mul(hi, w0);
                    return grp == 0 ? f64_add(lo, t) : f64_sub(lo, t);
                } else {
                    const uint64_t t = shoup_lazy(hi, w0.w, w0.wp, q);
                    return grp == 0 ? lo + t : lo - t + ar.q2;
                }
            },
            [&](uint32_t p, val a, val b) {
                if (h == 0) {
                    const auto a0 = M::load_key(p0 + p), a1 = M::load_key(p0 + p + 1);
                    const auto b0 = M::load_key(p1 + p), b1 = M::load_key(p1 + p + 1);
                    *reinterpret_cast<u64x2 *>(c0 + p) =
                        u64x2{M::bits(ar.mul_key(a, a0)), M::bits(ar.mul_key(b, a1))};
                    *reinterpret_cast<u64x2 *>(c1 + p) =
                        u64x2{M::bits(ar.mul_key(a, b0)), M::bits(ar.mul_key(b, b1))};
                } else {
                    const u64x2 t = *reinterpret_cast<const u64x2 *>(cc + p);
                    *reinterpret_cast<u64x2 *>(cc + p) =
                        u64x2{ar.canon_sum(a, M::from_bits(t.x)), ar.canon_sum(b, M::from_bits(t.y))};
                }
            },
            gsync);
        gsync();   // last-phase readers of this half are done before phase 0 writes
    }
    __syncthreads();
}

// The same for N = 2 * 2^LOGB (N = 2^14 with LOGB = 13): the thread block is
// two groups of threads, each of which transforms one half of the limb as a
// sub-block of the long transform on its own schedule (named barriers), so
// that one group's barrier and memory waits overlap the other's arithmetic.
// The stage that pairs the two halves is done on the way in, where both are at
// hand.
template <class L, int V>
__global__ void __launch_bounds__(2 * L::NT / V, 1)
encrypt_fused2_kernel(const __grid_constant__ CtxDev c, const KeysDev k, const float *sel, int64_t *mscr,
                      uint32_t t0, uint64_t seed, uint32_t client, uint64_t *ct, uint32_t T) {
    using LF = Lay<L::LOGB, 3>;                      // the slot transform of the ring (n = half a limb)
    static_assert(LF::NT == 2 * L::NT / V, "the encoder is played by the whole block");
    extern __shared__ __align__(128) uint64_t sm[];
    constexpr uint32_t H = 1u << L::LOGB, B = 2 * H;       // half and whole limb
    constexpr uint32_t GT = L::NT / V, RT = 2 * GT;        // threads per group, per block
    int8_t *su = reinterpret_cast<int8_t *>(sm + B);
    int8_t *se0 = su + B, *se1 = se0 + B;
    const uint32_t tid = threadIdx.x;
    __shared__ GaussTables gt_tab;
    gauss_tables_load(gt_tab, c.gauss, tid, blockDim.x);

    const uint64_t units = (uint64_t)T * c.L;
    const uint32_t u_begin = (uint32_t)(units * blockIdx.x / gridDim.x);
    const uint32_t u_end = (uint32_t)(units * (blockIdx.x + 1) / gridDim.x);
    const size_t cstride = (size_t)c.L * B;
    int64_t *mblk = mscr + (size_t)blockIdx.x * B;   // this block's encoded message (stays in L2)
    uint32_t sampled = 0xffffffffu;
    for (uint32_t unit = u_begin; unit < u_end; unit++) {
        const uint32_t tl = unit / c.L, j = unit % c.L;
        if (tl != sampled) {
            sampled = tl;
            const uint32_t t = t0 + tl;
            __syncthreads();
            for (uint32_t b = tid; b < B / 4; b += RT) {
                u32x4 w = stream_block(seed, b, t, client, TAG_ENC_U);
                char4 v = make_char4((signed char)ternary_from_word(w.x), (signed char)ternary_from_word(w.y),
                                     (signed char)ternary_from_word(w.z), (signed char)ternary_from_word(w.w));
                *reinterpret_cast<char4 *>(su + bswz(4 * b)) = v;
            }
            for (uint32_t b = tid; b < B / 2; b += RT) {
                const int2 a = gauss_pair(gt_tab, seed, b, t, client, TAG_ENC_E0), e = gauss_pair(gt_tab, seed, b, t, client, TAG_ENC_E1);
                *reinterpret_cast<char2 *>(se0 + bswz(2 * b)) = make_char2((signed char)a.x, (signed char)a.y);
                *reinterpret_cast<char2 *>(se1 + bswz(2 * b)) = make_char2((signed char)e.x, (signed char)e.y);
            }
            // the ciphertext's message: slot transform, scaling and rounding in the limb buffer
            if (encode_in_block<LF>(c, sel + (size_t)tl * H, sm, mblk)) atomicOr(c.status, STATUS_RANGE);
        }
        const LimbDev &lb = c.limb[j];
        uint64_t *cbase = ct + (((size_t)tl * 2 + 0) * c.L + j) * B;
        FEDHE_FOR_ARITH_SEL(lb, (encrypt_unit2<M_, L, V>(lb, k.pk0_hat + (size_t)j * B, k.pk1_hat + (size_t)j * B, sm, su,
                                                     se0, mblk, cbase, cstride)));
    }
}

// Long rings: kernels over the 2^A x 2^13 view of a limb.

template <class M, uint32_t A>
__device__ __forceinline__ void enc_outer_sample_limb(const LimbDev &lb, const int (&u)[1u << A][2], uint64_t *p,
                                                      uint32_t B) {
    constexpr uint32_t rows = 1u << A;
    const auto t = LimbOf<M>::args(lb, true, 0, 0);
    typename M::val x[rows], y[rows];
#pragma unroll
    for (uint32_t a = 0; a < rows; a++) {
        x[a] = t.m.small(u[a][0]);
        y[a] = t.m.small(u[a][1]);
    }
    outer_forward<A>(x, y, t);
#pragma unroll
    for (uint32_t a = 0; a < rows; a++)
        *reinterpret_cast<u64x2 *>(p + (size_t)a * B) = u64x2{M::bits(x[a]), M::bits(y[a])};
}

// one thread per pair of neighbouring columns of one ciphertext, all limbs: draws u and runs the outer forward stages;
// the limbs of ciphertext tl go to dst + tl * ct_stride
template <uint32_t A>
__global__ void __launch_bounds__(256)
enc_outer_sample_kernel(const __grid_constant__ CtxDev c, uint32_t t0, uint64_t seed, uint32_t client,
                        uint64_t *dst, size_t ct_stride, size_t total) {
    size_t g = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (g >= total) return;
    const uint32_t B = 1u << c.LOGB, half = B >> 1;
    constexpr uint32_t rows = 1u << A;
    const uint32_t col = (uint32_t)(g % half) * 2;
    const size_t tl = g / half;
    int u[rows][2];
#pragma unroll
    for (uint32_t a = 0; a < rows; a++) {
        const uint32_t i = a * B + col;               // even: both columns share a Philox block
        const u32x4 w = stream_block(seed, i >> 2, t0 + (uint32_t)tl, client, TAG_ENC_U);
        u[a][0] = ternary_from_word((i & 2) ? w.z : w.x);
        u[a][1] = ternary_from_word((i & 2) ? w.w : w.y);
    }
#pragma unroll 1
    for (uint32_t j = 0; j < c.L; j++) {
        const LimbDev &lb = c.limb[j];
        uint64_t *p = dst + tl * ct_stride + (size_t)j * c.N + col;   // limb j of ciphertext tl
        FEDHE_FOR_ARITH(lb, (enc_outer_sample_limb<M_, A>(lb, u, p, B)));
    }
}

// one thread block per (ciphertext, limb, block): forward block transform of u, products with both halves
// of the public key on the way out
template <class M, class L, int V, bool ACC>
__device__ __forceinline__ void enc_block_forward(const CtxDev &c, const LimbDev &lb, uint64_t *sm, uint32_t blk,
                                                  const tw_t *p0, const tw_t *p1, const uint64_t *u,
                                                  uint64_t *c0, uint64_t *c1) {
    using val = typename M::val;
    const auto a = LimbOf<M>::args(lb, true, c.A, blk);
    const M &ar = a.m;
    smem_ntt_forward<L, V>(
        sm, threadIdx.x, a, [&](uint32_t i) { return M::from_bits(u[i]); },
        [&](uint32_t p, val x, val y) {
            const auto a0 = M::load_key(p0 + p), a1 = M::load_key(p0 + p + 1);
            const auto b0 = M::load_key(p1 + p), b1 = M::load_key(p1 + p + 1);
            u64x2 v0, v1;
            if constexpr (ACC) {       // the slots hold canonical residues to add to
                v0 = *reinterpret_cast<const u64x2 *>(c0 + p);
                v1 = *reinterpret_cast<const u64x2 *>(c1 + p);
                v0.x = ar.canon_add(ar.mul_key(x, a0), v0.x);
                v0.y = ar.canon_add(ar.mul_key(y, a1), v0.y);
                v1.x = ar.canon_add(ar.mul_key(x, b0), v1.x);
                v1.y = ar.canon_add(ar.mul_key(y, b1), v1.y);
            } else {
                v0.x = ar.to_residue(ar.mul_key(x, a0));
                v0.y = ar.to_residue(ar.mul_key(y, a1));
                v1.x = ar.to_residue(ar.mul_key(x, b0));
                v1.y = ar.to_residue(ar.mul_key(y, b1));
            }
            *reinterpret_cast<u64x2 *>(c0 + p) = v0;
            *reinterpret_cast<u64x2 *>(c1 + p) = v1;
        });
}

// ACC = false: u comes from the c1 slot and the products replace both slots;
// ACC = true: u comes from `ubuf` ([T][L][N]) and the products are added to the slots
template <class L, int V, bool ACC>
__global__ void __launch_bounds__(L::NT / V, (L::NT / V) <= 512 ? 2 : 1)
enc_block_forward_kernel(const __grid_constant__ CtxDev c, const KeysDev k, const uint64_t *ubuf, uint64_t *ct) {
    extern __shared__ __align__(128) uint64_t sm[];
    uint32_t b = blockIdx.x;
    const uint32_t blk = b & ((1u << c.A) - 1u);
    b >>= c.A;
    const uint32_t j = b % c.L;
    const size_t tl = b / c.L;
    const LimbDev &lb = c.limb[j];
    const size_t off = ((size_t)blk << L::LOGB);
    uint64_t *c0 = ct + ((tl * 2 + 0) * c.L + j) * c.N + off;
    uint64_t *c1 = ct + ((tl * 2 + 1) * c.L + j) * c.N + off;
    const uint64_t *u = ACC ? ubuf + (tl * c.L + j) * c.N + off : c1;
    const tw_t *p0 = k.pk0_hat + (size_t)j * c.N + off, *p1 = k.pk1_hat + (size_t)j * c.N + off;
    FEDHE_FOR_ARITH(lb, (enc_block_forward<M_, L, V, ACC>(c, lb, sm, blk, p0, p1, u, c0, c1)));
}

// residues of e0 + m into the c0 slots and
// of e1 into the c1 slots; one thread per pair of neighbouring coefficients
__global__ void __launch_bounds__(256)
enc_fill_errors_kernel(const __grid_constant__ CtxDev c, const int64_t *m, uint32_t t0, uint64_t seed,
                       uint32_t client, uint64_t *ct, size_t total) {
    __shared__ GaussTables gt;
    gauss_tables_load(gt, c.gauss, threadIdx.x, blockDim.x);
    __syncthreads();
    const size_t g = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (g >= total) return;
    const uint32_t pairs = c.N >> 1;
    const uint32_t b = (uint32_t)(g % pairs), i = 2 * b;   // one Philox block per pair
    const size_t tl = g / pairs;
    const uint32_t t = t0 + (uint32_t)tl;
    const int2 e0 = gauss_pair(gt, seed, b, t, client, TAG_ENC_E0), e1 = gauss_pair(gt, seed, b, t, client, TAG_ENC_E1);
    const longlong2 mm = *reinterpret_cast<const longlong2 *>(m + tl * c.N + i);
    const int64_t ax = mm.x + e0.x, ay = mm.y + e0.y;
    const int ex = e1.x, ey = e1.y;
    for (uint32_t j = 0; j < c.L; j++) {
        const LimbDev &lb = c.limb[j];
        const uint64_t q = lb.q;
        *reinterpret_cast<u64x2 *>(ct + ((tl * 2 + 0) * c.L + j) * c.N + i) =
            u64x2{signed_residue(ax, q, lb.mu), signed_residue(ay, q, lb.mu)};
        *reinterpret_cast<u64x2 *>(ct + ((tl * 2 + 1) * c.L + j) * c.N + i) =
            u64x2{small_residue(ex, q), small_residue(ey, q)};
    }
}

template <class M, uint32_t A>
__device__ __forceinline__ void enc_outer_inverse_add_limb(const LimbDev &lb, uint64_t *p, uint32_t B,
                                                           const int64_t (&add)[1u << A][2]) {
    constexpr uint32_t rows = 1u << A;
    const uint64_t q = lb.q;
    const auto t = LimbOf<M>::args(lb, false, 0, 0);
    typename M::val x[rows], y[rows];
#pragma unroll
    for (uint32_t a = 0; a < rows; a++) {
        const u64x2 v = *reinterpret_cast<const u64x2 *>(p + (size_t)a * B);
        x[a] = M::from_bits(v.x);
        y[a] = M::from_bits(v.y);
    }
    outer_inverse<A>(x, y, t, LimbOf<M>::ninv(lb), LimbOf<M>::wn(lb));
#pragma unroll
    for (uint32_t a = 0; a < rows; a++) {
        u64x2 o;
        o.x = t.m.canon_add(x[a], signed_residue(add[a][0], q, lb.mu));
        o.y = t.m.canon_add(y[a], signed_residue(add[a][1], q, lb.mu));
        *reinterpret_cast<u64x2 *>(p + (size_t)a * B) = o;
    }
}

// one thread per pair of neighbouring columns of one ciphertext: for each
// component draws its error terms once (e0 + m, then e1), then finishes every limb
template <uint32_t A>
__global__ void __launch_bounds__(256, A == 3 ? 2 : 4)
enc_outer_inverse_add_kernel(const __grid_constant__ CtxDev c, const int64_t *m, uint32_t t0, uint64_t seed,
                             uint32_t client, uint64_t *ct, size_t total) {
    __shared__ GaussTables gt;
    gauss_tables_load(gt, c.gauss, threadIdx.x, blockDim.x);
    __syncthreads();
    size_t g = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (g >= total) return;
    const uint32_t B = 1u << c.LOGB, half = B >> 1;
    constexpr uint32_t rows = 1u << A;
    const uint32_t col = (uint32_t)(g % half) * 2;
    const size_t tl = g / half;
    const uint32_t t = t0 + (uint32_t)tl;
#pragma unroll 1
    for (uint32_t comp = 0; comp < 2; comp++) {
        int64_t add[rows][2];                          // e0 + m, or e1
#pragma unroll
        for (uint32_t a = 0; a < rows; a++) {
            const uint32_t i = a * B + col;           // one Philox block per pair of coefficients
            const int2 e = gauss_pair(gt, seed, i >> 1, t, client, comp == 0 ? TAG_ENC_E0 : TAG_ENC_E1);
            add[a][0] = e.x;
            add[a][1] = e.y;
            if (comp == 0) {
                const longlong2 mm = *reinterpret_cast<const longlong2 *>(m + tl * c.N + i);
                add[a][0] += mm.x;
                add[a][1] += mm.y;
            }
        }
#pragma unroll 1
        for (uint32_t j = 0; j < c.L; j++) {
            const LimbDev &lb = c.limb[j];
            uint64_t *p = ct + ((tl * 2 + comp) * c.L + j) * c.N + col;
            FEDHE_FOR_ARITH(lb, (enc_outer_inverse_add_limb<M_, A>(lb, p, B, add)));
        }
    }
}

// shared memory of a block of the fused kernels: the limb and three one-byte sample arrays
static size_t fused_smem(const CtxDev &c) { return ((size_t)c.N << 3) + 3 * (size_t)c.N; }

// The fused kernels run one block per SM for N = 2^14 and two for N = 2^13 (what
// their shared memory allows); every block owns N words of message scratch.
size_t encrypt_fused_blocks(const CtxDev &c, int n_sm) {
    const size_t per_sm = (size_t)(227 * 1024) / fused_smem(c);
    return (size_t)n_sm * (per_sm ? per_sm : 1);
}

template <class L, int V, bool TWO_GROUPS>
static cudaError_t launch_encrypt_fused(const CtxDev &c, const KeysDev &k, const float *sel, int64_t *mscr,
                                        int n_sm, uint32_t t0, size_t T, uint64_t seed, uint32_t client,
                                        uint64_t *ct, cudaStream_t s) {
    const size_t smem = fused_smem(c);
    auto kern = TWO_GROUPS ? encrypt_fused2_kernel<L, V> : encrypt_fused_kernel<L, V>;
    cudaError_t e;
    if ((e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem))) return e;
    size_t grid = encrypt_fused_blocks(c, n_sm);                     // fewer if there is less work
    if (grid > T * c.L) grid = T * c.L;
    kern<<<(unsigned)grid, (TWO_GROUPS ? 2 : 1) * L::NT / V, smem, s>>>(c, k, sel, mscr, t0, seed, client, ct,
                                                                        (uint32_t)T);
    return FEDHE_LAUNCHED();
}

// launches the block forward kernel of the long-ring paths
template <bool ACC>
static cudaError_t launch_enc_block_forward(const CtxDev &c, const KeysDev &k, const uint64_t *ubuf, size_t T,
                                            uint64_t *ct, cudaStream_t s) {
    using L = WLay<13>;                                 // long rings are cut into 2^13 blocks
    constexpr int V = 2;
    const size_t smem = sizeof(uint64_t) << L::LOGB;
    auto kern = enc_block_forward_kernel<L, V, ACC>;
    cudaError_t e;
    if ((e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem))) return e;
    kern<<<(unsigned)((T * c.L) << c.A), L::NT / V, smem, s>>>(c, k, ubuf, ct);
    return FEDHE_LAUNCHED();
}

size_t encrypt_ntt_work_bytes(const CtxDev &c, int n_sm, size_t T) {
    if (c.A == 0) return encrypt_fused_blocks(c, n_sm) * c.N * sizeof(int64_t);
    // long rings: the encoded messages, the encoder's complex buffer and the transform of u
    return (2 + (size_t)c.L) * T * c.N * sizeof(uint64_t);
}

// Transform-domain wire format: the same ciphertext with every limb polynomial
// stored as its negacyclic transform.  N <= 2^14: the fused kernels with three
// forward transforms per limb.  Longer rings: the error terms go into the
// ciphertext slots and are transformed there; u is transformed in the work
// buffer `ubuf` ([T][L][N]) and its key products are added on the way out.
cudaError_t launch_encrypt_ntt(const CtxDev &c, const KeysDev &k, const float *sel, void *work, int n_sm,
                               uint32_t t0, size_t T, uint64_t seed, uint32_t client, uint64_t *ct,
                               cudaStream_t s) {
    if (T == 0) return cudaSuccess;
    int64_t *m = static_cast<int64_t *>(work);
    if (c.A == 0) {
        if (c.LOGB == 13)
            return launch_encrypt_fused<WLay<13>, 2, false>(c, k, sel, m, n_sm, t0, T, seed, client, ct, s);
        return launch_encrypt_fused<WLay<13>, 2, true>(c, k, sel, m, n_sm, t0, T, seed, client, ct, s);
    }
    cudaError_t e;
    uint64_t *ubuf = reinterpret_cast<uint64_t *>(m + 2 * T * c.N);
    if ((e = launch_encode(c, sel, T, reinterpret_cast<double2 *>(m + T * c.N), m, s))) return e;
    const size_t LN = (size_t)c.L * c.N;
    const size_t pairs = T * (size_t)(c.N >> 1);
    enc_fill_errors_kernel<<<blocks_for(pairs, 256), 256, 0, s>>>(c, m, t0, seed, client, ct, pairs);
    if ((e = FEDHE_LAUNCHED())) return e;
    if ((e = launch_ntt(c, true, ct, 2 * T, LN, 0, c.L, s))) return e;
    const size_t cols = T * ((size_t)1 << (c.LOGB - 1));
    FEDHE_FOR_A(c, (enc_outer_sample_kernel<A_><<<blocks_for(cols, 256), 256, 0, s>>>(c, t0, seed, client, ubuf, LN,
                                                                                     cols)));
    if ((e = FEDHE_LAUNCHED())) return e;
    return launch_enc_block_forward<true>(c, k, ubuf, T, ct, s);
}

// Coefficient format on the longest ring by passes over the ciphertext itself, which is the work space: (1) draw u
// and run the outer forward stages into the c1 slots; (2) block transforms of the c1 slots whose last phase
// writes both products u^ pk0^ -> c0 and u^ pk1^ -> c1; (3) inverse block transforms of all slots; (4) outer
// inverse stages fused with the error and message terms.  `work`: the encoded messages and the encoder's complex buffer.
//
// A limb of N = 2^16 is eight blocks of the complex transforms, which one thread block computes one after the other, and what a
// number of ciphertexts takes rises in steps with the rounds of clusters; the passes take the same for every ciphertext, less for limbs
// below 2^46.  So with 60-bit limbs the passes are faster for few ciphertexts, and with 45-bit ones but for some counts just short of
// a round, and again for many.  Measured (us, passes and transforms):
//   two 60-bit limbs: 10, 24, 40, 92, 600 ciphertexts   143 214, 216 224, 341 333, 653 546, 3961 2870
//   eight: 3, 5, 18, 40   180 177, 214 173, 452 478, 986 642;      four of 45 bits: 10, 31, 40, 92, 600   147 185, 298 298, 394 439, 761 824, 4608 4919
//   twelve of 45 bits: 3, 10, 31, 92, 300   165 179, 300 407, 718 732, 1949 2141, 6166 6578
// (by transforms that have got 4 to 9 % faster since, with two 60-bit limbs 24 and 600 ciphertexts take 197 and 2770 now; the passes are as they were).
// The passes by the line through these (up to 20 % low short of a whole wave of their thread blocks, hence 4 to 7 % in their favour),
// the transforms by the cost of their plan.
bool encrypt_by_passes(const CtxDev &c, size_t T) {
    if (c.logN < 16) return false;
    if (T > PASSES_KNOWN) return c.passes_most > PASSES_KNOWN;
    double fixed = 40.0, per_ct = 1.5, favour = 1.04;
    for (uint32_t j = 0; j < c.L; j++) {
        const bool in_doubles = c.limb[j].fwd_d != nullptr;
        fixed += in_doubles ? 4.0 : 6.0 + 20.0 / c.L;
        per_ct += in_doubles ? 1.54 : 2.48;
        if (in_doubles) favour = 1.07;
    }
    return fixed + per_ct * (double)T < favour * enc_transforms_us(c, T);
}
// The largest number of ciphertexts that goes by passes: up to PASSES_KNOWN by the rule, beyond like the last counts before.
uint32_t passes_most(const CtxDev &c) {
    if (c.logN < 16) return 0;
    uint32_t T = PASSES_KNOWN;
    while (T && !encrypt_by_passes(c, T)) T--;
    return T > PASSES_KNOWN - 64 ? UINT32_MAX : T;
}
// what the passes need for any number of ciphertexts up to T
size_t encrypt_passes_work_bytes(const CtxDev &c, size_t T) {
    return 2 * (T < c.passes_most ? T : (size_t)c.passes_most) * c.N * sizeof(uint64_t);
}
cudaError_t launch_encrypt_passes(const CtxDev &c, const KeysDev &k, const float *sel, void *work, uint32_t t0, size_t T,
                                  uint64_t seed, uint32_t client, uint64_t *ct, cudaStream_t s) {
    if (T == 0) return cudaSuccess;
    int64_t *m = static_cast<int64_t *>(work);
    cudaError_t e;
    if ((e = launch_encode(c, sel, T, reinterpret_cast<double2 *>(m + T * c.N), m, s))) return e;
    const size_t cols = T * ((size_t)1 << (c.LOGB - 1));      // pairs of columns
    const size_t LN = (size_t)c.L * c.N;
    enc_outer_sample_kernel<3><<<blocks_for(cols, 256), 256, 0, s>>>(c, t0, seed, client, ct + LN, 2 * LN, cols);
    if ((e = FEDHE_LAUNCHED())) return e;
    if ((e = launch_enc_block_forward<false>(c, k, nullptr, T, ct, s))) return e;
    if ((e = launch_ntt_inner(c, false, ct, 2 * T, LN, 0, c.L, s))) return e;
    enc_outer_inverse_add_kernel<3><<<blocks_for(cols, 256), 256, 0, s>>>(c, m, t0, seed, client, ct, cols);
    return FEDHE_LAUNCHED();
}

}  // namespace fedhe

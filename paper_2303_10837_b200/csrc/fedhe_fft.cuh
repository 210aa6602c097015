// Exact products of a small polynomial and a large one by complex transforms.
//
// Encryption and decryption multiply, in Z[X]/(X^N + 1), a ternary polynomial
// (u or s) by a polynomial with coefficients up to 2^61 (a half of the public
// key, or c1).  Every number-theoretic transform of such a limb costs about 26
// slots of the multiply / double-precision pipe per butterfly on a 60-bit prime
// (8 or 9 on a prime below 2^46), and one product takes one or two of them per
// limb and direction.  Here the large operand is cut into pieces, p = sum_i p_i 2^(s_i),
// every product p_i * t is computed by a complex
// transform of n = N/2 points in fp64 and rounded: a coefficient z_k =
// a_k + i a_(k+n) turns the negacyclic ring of degree N into C[X]/(X^n - i).
// A butterfly is 6 fused multiply-adds and there are half as many of them, the
// transform of the ternary operand is shared by all limbs, and neither
// modular products nor conditional subtractions occur: 395 k slots per piece
// at N = 2^14 against 3.0 M per 60-bit transform.
//
// The rounded coefficients are the exact integers.  Let e = 2^-53.
//   One butterfly (s, d) = (x + w y, x - w y) is evaluated as t = x - w_i y',
//   s = t + w_r y (two roundings per component) and d = 2 x - s (one more).  Its
//   error is at most e(|t| + |s|) in s and e(|t| + |s| + |d|) in d, and with the
//   twiddle's own rounding (each component at most 2^-54 off) at most
//   3.8 e times the norm of the butterfly's output.
//   * Forward transforms: in the 2-norm the errors of the levels add up to
//     3.8 e levels * sqrt(n) ||t||_2, and likewise for the pieces (the key
//     tables are made by the same code).
//   * Product: |error| <= 2.3 e |t^||p^| per point; by Cauchy-Schwarz the sum over the points
//     of all the errors so far is at most (7.6 levels + 2.3) e * n ||t||_2 ||p_i||_2.
//   * Inverse: an output depends, at every level, on nodes that are sums over
//     disjoint sets of inputs, so a level adds at most 3.8 e (1/n) sum |z^_j|
//     <= 3.8 e ||t||_2 ||p_i||_2 to it.
//   * The twiddles that are made by products with constants (4 e off each), the
//     untwisting factor in its two parts: 20 e together.
// With ||t||_2 <= sqrt(N), ||p_i||_2 <= 2^(b-1) sqrt(N) for pieces of b bits:
//   |error| <= (11.4 levels + 23) 2^-53 N 2^(b-1)
// = 0.17 for N = 2^14 (13 levels, b = 30), 0.36 for N = 2^15 (14, 30), and
// 0.38 for N = 2^16 (15, 29): below 1/2, whatever the two operands are.
// fft_sure_bits() evaluates this bound; decryption, whose c1 comes from outside,
// cuts by it.
//
// In encryption both operands are the library's own random draws (u ternary, the
// public key uniform), so the coefficients and the rounding errors, sums of
// some 10^6 independent ones, stay near their standard deviations, which are
// about sqrt(N) times smaller than the bounds above.  For pieces of b bits
//   sd(error) <= 1.3 sqrt(levels) 2^-53 * sd(product),  sd(product) = sqrt(N / 18) 2^b
// (1.2 to 1.3 measured on every ring).  fft_wide_bits() keeps 24 standard
// deviations below 1/2, a chance of a wrong coefficient under 2^-400: 40 bits at N = 2^14, so that a
// 40-bit limb is one piece and a 60-bit one is two.
//
// The tests play both directions on the host, thread by thread.
#pragma once

#include "fedhe_device.cuh"

namespace fedhe {

struct cpx { double re, im; };
struct alignas(16) root_t { double re, im; };      // a table entry

constexpr int FFT_MAX_PIECES = 3;

// largest pieces whose rounding error stays below 0.45 for any operands
inline int fft_sure_bits(int logN) {
    for (int b = 30; b > 1; b--) {
        const double err = (11.4 * (logN - 1) + 23.0) * (double)(1ull << (logN + b - 1)) / 9007199254740992.0;
        if (err < 0.45) return b;
    }
    return 0;
}
// standard deviation of the error for pieces of b bits of a random operand
inline double fft_error_sd(int logN, int b) {
    return 1.3 * sqrt((double)(logN - 1) * (double)(1ull << logN) / 18.0) * (double)(1ull << b) / 9007199254740992.0;
}
// largest such pieces with 24 standard deviations below 1/2
inline int fft_wide_bits(int logN) {
    int b = 44;
    while (24.0 * fft_error_sd(logN, b) >= 0.5) b--;
    return b;
}

// Widest random piece whose product stays below 2^(t - 1).  A coefficient is a sum of N independent terms u_k p_k,
// strictly sub-Gaussian with variance 2^(2 width) / 18 each, so the chance of a larger one is at most
// 2 exp(-9 2^(2 t - 2) / (N 2^(2 width))); `least` is what the exponent has to reach.
inline int fft_random_bits(int logN, int t, double least) {
    int w = 0;
    while (ldexp(9.0, 2 * t - 2 - logN - 2 * (w + 1)) >= least) w++;
    return w;
}
// `least` for the 16-bit products of two limbs' low pieces, and for 32-bit ones
constexpr double FFT_PAIR_EXPONENT = 72.0, FFT_NARROW_EXPONENT = 95.0;

// ---- geometry ------------------------------------------------------------------
//
// A block of NB = 2^12 points is transformed by NT = 256 threads with 16 points
// in registers.  Three layouts, a third of the position bits each:
//   A: reg {0..3}  lane {4..8}     warp {9..11}      position 16 tid + r
//   B: reg {4..7}  lane {0..3, 8}  warp {9..11}
//   C: reg {8..11} lane {0..4}     warp {5..7}       position tid + NT r
// A <-> B stays inside a warp (its own 512 points of the buffer, a warp-level
// barrier), B <-> C crosses the block: 12 stages, two exchanges through shared memory.
// A transform of n = 2^(12 + CL) points is cut into R = 2^CL such blocks, which a
// thread block does one after the other; the CL stages between them are done where a
// thread has an element of every block at hand.
//
// Forward (coefficients in order -> values, bit-reversed): level l splits
// X^m = c^2 into X^(m/2) = +-c, so its twiddle depends on the block only:
// fwd[2^l + block] (and, for the last four levels, a copy in the threads' order behind it).  Inverse (values, bit-reversed -> coefficients): decimation
// in time with the twiddles exp(-2 pi i j / len), then the factor omega^-k,
// omega = exp(i pi / N): omega^-tid goes in with the twiddles of the last four
// stages, the rest of it is a constant of the register.
struct FftLay {
    static constexpr int LB = 12, NB = 1 << LB, NT = NB / 16;
    // words (of 16 bytes) of a warp's part of the buffer
    static HD uint32_t a_word(uint32_t lane, int r) { return lane * 16 + ((uint32_t)r ^ (lane & 7u)); }
    static HD uint32_t b_word(uint32_t lane, int r) {
        return (lane >> 4) * 256 + (uint32_t)r * 16 + ((lane & 15u) ^ ((uint32_t)r & 7u));
    }
    // words of the exchange between B and C
    static HD uint32_t bc_word(uint32_t lane, int r) { return (lane >> 4) * 256 + (uint32_t)r * 16 + (lane & 15u); }
};

// Inverse tables, copied into shared memory once per thread block (entries of 16 bytes):
//   [0, 128)      layout B: 8 runs of 16, indexed by position bits 0..3
//   then 5 + CL runs of NT: omega^-tid, the four stages of layout C, the CL stages between blocks
//   then 16 runs of TURNS for the registers' constants of the stages between blocks and of omega^-k
template <int CL>
struct FftTab {
    static constexpr int C = 128, NT = FftLay::NT, BETWEEN = C + 5 * NT, TURN = BETWEEN + CL * NT,
                         TURNS = (CL == 0 ? 0 : 1 << (CL > 0 ? CL - 1 : 0)) + (1 << CL), WORDS = TURN + 16 * TURNS;
};

// ---- butterflies -----------------------------------------------------------------

HD void fft_bf(cpx &x, cpx &y, double wr, double wi) {
    const double sr = f64_fma(wr, y.re, f64_fma(-wi, y.im, x.re)), si = f64_fma(wr, y.im, f64_fma(wi, y.re, x.im));
    y.re = f64_fma(2.0, x.re, -sr);
    y.im = f64_fma(2.0, x.im, -si);
    x.re = sr;
    x.im = si;
}
HD void fft_bf_one(cpx &x, cpx &y) {                       // w = 1
    const cpx u = x, v = y;
    x.re = f64_add(u.re, v.re);
    x.im = f64_add(u.im, v.im);
    y.re = f64_sub(u.re, v.re);
    y.im = f64_sub(u.im, v.im);
}
HD void fft_bf_mi(cpx &x, cpx &y) {                        // w = -i
    const cpx u = x, v = y;
    x.re = f64_add(u.re, v.im);
    x.im = f64_sub(u.im, v.re);
    y.re = f64_sub(u.re, v.im);
    y.im = f64_add(u.im, v.re);
}
HD cpx cpx_mul(cpx a, double wr, double wi) {
    return cpx{f64_fma(-wi, a.im, f64_mul(wr, a.re)), f64_fma(wi, a.re, f64_mul(wr, a.im))};
}

// cos(pi k / 16), |k| <= 16, to the nearest double.  In unrolled device code an entry is an operand
// in constant memory, where a literal would cost two moves at every use.
#define FEDHE_COS_PI16 {1.0, 0.9807852804032304, 0.9238795325112867, 0.8314696123025452, 0.7071067811865476,  \
                        0.5555702330196022, 0.3826834323650898, 0.19509032201612828, 0.0}
#if defined(__CUDACC__)
static __constant__ double c_cos_pi16[9] = FEDHE_COS_PI16;
#endif
HD double cos_pi16(int k) {
#if !defined(__CUDA_ARCH__)
    constexpr double c_cos_pi16[9] = FEDHE_COS_PI16;
#endif
    k = k < 0 ? -k : k;
    return k <= 8 ? c_cos_pi16[k] : -c_cos_pi16[16 - k];
}
HD double sin_pi16(int k) { return cos_pi16(8 - k); }

// ---- inverse -----------------------------------------------------------------------

// stages 1..4 in layout A: every twiddle is a constant exp(-i pi m / 2^I)
template <int I>
HD void inv_stage_const(cpx (&x)[16]) {
#pragma unroll
    for (int r = 0; r < 16; r++) {
        if (r & (1 << I)) continue;
        const int m = r & ((1 << I) - 1);
        cpx &a = x[r], &b = x[r | (1 << I)];
        if (m == 0) fft_bf_one(a, b);
        else if (2 * m == (1 << I)) fft_bf_mi(a, b);
        else fft_bf(a, b, cos_pi16(m << (4 - I)), -sin_pi16(m << (4 - I)));
    }
}
HD void inv_phase_a(cpx (&x)[16]) {
    inv_stage_const<0>(x);
    inv_stage_const<1>(x);
    inv_stage_const<2>(x);
    inv_stage_const<3>(x);
}

// butterflies of stage I of a phase whose lower register has the low bits m (mod
// 2^I): twiddle w, and w (-i) for the registers half a period further
template <int I>
HD void inv_group(cpx (&x)[16], int m, double wr, double wi) {
#pragma unroll
    for (int r = 0; r < 16; r++) {
        if (r & (1 << I)) continue;
        const int low = r & ((1 << I) - 1);
        if (low == m) fft_bf(x[r], x[r | (1 << I)], wr, wi);
        else if (I >= 1 && low == m + (1 << (I >= 1 ? I - 1 : 0))) fft_bf(x[r], x[r | (1 << I)], wi, -wr);
    }
}

// stages 5..8 in layout B; j0 = position bits 0..3
HD void inv_phase_b(cpx (&x)[16], const root_t *tb, uint32_t j0) {
    const root_t *t = tb + j0;
    inv_group<0>(x, 0, t[0].re, t[0].im);
    inv_group<1>(x, 0, t[16].re, t[16].im);
    inv_group<2>(x, 0, t[32].re, t[32].im);
    inv_group<2>(x, 1, t[48].re, t[48].im);
#pragma unroll
    for (int m = 0; m < 4; m++) inv_group<3>(x, m, t[64 + 16 * m].re, t[64 + 16 * m].im);
}

// the last four stages in layout C with omega^-tid: the inputs of the first stage that meet no
// twiddle take the factor by a product, the others with their twiddle
HD void inv_phase_c(cpx (&x)[16], const root_t *tc, uint32_t tid) {
    constexpr int NT = FftLay::NT;
    const root_t *t = tc + tid;
    {
        const double tr = t[0].re, ti = t[0].im;
        const cpx w = cpx_mul(cpx{t[NT].re, t[NT].im}, tr, ti);
#pragma unroll
        for (int r = 0; r < 16; r += 2) {
            x[r] = cpx_mul(x[r], tr, ti);
            fft_bf(x[r], x[r + 1], w.re, w.im);
        }
    }
    inv_group<1>(x, 0, t[2 * NT].re, t[2 * NT].im);
    {
        const cpx w = {t[3 * NT].re, t[3 * NT].im};
        inv_group<2>(x, 0, w.re, w.im);
        const cpx v = cpx_mul(w, cos_pi16(4), -sin_pi16(4));
        inv_group<2>(x, 1, v.re, v.im);
    }
    {
        const cpx w = {t[4 * NT].re, t[4 * NT].im};
        inv_group<3>(x, 0, w.re, w.im);
#pragma unroll
        for (int m = 1; m < 4; m++) {
            const cpx v = cpx_mul(w, cos_pi16(2 * m), -sin_pi16(2 * m));
            inv_group<3>(x, m, v.re, v.im);
        }
    }
}

// ---- forward -----------------------------------------------------------------------

HD cpx fft_root(const root_t *p) {
#if defined(__CUDA_ARCH__)
    const double2 v = __ldg(reinterpret_cast<const double2 *>(p));
    return cpx{v.x, v.y};
#else
    return cpx{p->re, p->im};
#endif
}

// Four levels on the registers, top bit first; root(i, g): the twiddle of group g (even) of level i.  The
// group after it has the same one times the imaginary unit.
template <class Root>
HD void fwd_phase4(cpx (&x)[16], const Root &root) {
#pragma unroll
    for (int i = 0; i < 4; i++) {
        const int bit = 3 - i;
#pragma unroll
        for (int g = 0; g < (1 << i); g += 2) {
            const cpx w = root(i, g);
#pragma unroll
            for (int k = 0; k < (1 << bit); k++) {
                const int r = (g << (4 - i)) + k;
                fft_bf(x[r], x[r + (1 << bit)], w.re, w.im);
                if (i > 0) fft_bf(x[r + (2 << bit)], x[r + (3 << bit)], -w.im, w.re);
            }
        }
    }
}
// index: the thread's block at the first level (2^l + block); the runs of the next levels follow by doubling
HD void fwd_phase4_at(cpx (&x)[16], const root_t *fwd, uint32_t index) {
    fwd_phase4(x, [&](int i, int g) { return fft_root(fwd + (index << i) + g); });
}
// the last phase of a block, whose eight twiddles per thread have a table in the threads' order: [8][NT] per block
constexpr int FFT_LAST = 8 * FftLay::NT;
HD void fwd_phase4_last(cpx (&x)[16], const root_t *last, uint32_t tid) {
    fwd_phase4(x, [&](int i, int g) { return fft_root(last + ((i == 0 ? 0 : 1 << (i - 1)) + g / 2) * FftLay::NT + tid); });
}

// ---- the stages between blocks ---------------------------------------------------------

// forward: v[a] = coefficient column + a NB -> v[b] = the column's value in block b
template <int CL>
HD void fft_outer_forward(cpx (&v)[1 << CL], const root_t *fwd) {
#pragma unroll
    for (int l = 0; l < CL; l++) {
        const int half = 1 << (CL - 1 - l);
#pragma unroll
        for (int g = 0; g < (1 << l); g++) {
            const cpx w = fft_root(fwd + (1 << l) + g);
#pragma unroll
            for (int k = 0; k < half; k++) fft_bf(v[2 * half * g + k], v[2 * half * g + k + half], w.re, w.im);
        }
    }
}

// the same for one block b: z mod (X^NB - rho_b), by the twiddles of the block's path with their signs
template <int CL>
struct OuterPath {
    cpx w[CL ? CL : 1];
    HD OuterPath(const root_t *fwd, uint32_t b) {
#pragma unroll
        for (int l = 0; l < CL; l++) {
            const uint32_t blk = b >> (CL - 1 - l);
            const cpx t = fft_root(fwd + (1u << l) + (blk >> 1));
            w[l] = (blk & 1u) ? cpx{-t.re, -t.im} : t;
        }
    }
    HD cpx apply(cpx (&z)[1 << CL]) const {
#pragma unroll
        for (int l = 0; l < CL; l++) {
            const int half = 1 << (CL - 1 - l);
#pragma unroll
            for (int k = 0; k < half; k++) {
                const cpx a = z[k + half];
                z[k] = cpx{f64_fma(w[l].re, a.re, f64_fma(-w[l].im, a.im, z[k].re)),
                           f64_fma(w[l].re, a.im, f64_fma(w[l].im, a.re, z[k].im))};
            }
        }
        return z[0];
    }
};

// inverse: v[b] = the value of column tid + NT r in block b -> v[a] = coefficient column + a NB, with
// what is missing of the factor omega^-k
template <int CL>
HD void fft_outer_inverse(cpx (&v)[1 << CL], const root_t *tab, uint32_t tid, uint32_t r) {
    using T = FftTab<CL>;
    constexpr int R = 1 << CL;
    const root_t *turn = tab + T::TURN + r * T::TURNS;
    int next = 0;
#pragma unroll
    for (int i = 0; i < CL; i++) {
        const root_t t = tab[T::BETWEEN + i * T::NT + tid];
#pragma unroll
        for (int a = 0; a < (i == 0 ? 1 : (1 << i) / 2); a++) {
            const cpx w = cpx_mul(cpx{t.re, t.im}, turn[next].re, turn[next].im);
            next++;
#pragma unroll
            for (int g = 0; g < R; g += 2 << i) {
                fft_bf(v[g + a], v[g + a + (1 << i)], w.re, w.im);
                if (i >= 1) {                                        // a quarter period further
                    const int q = g + a + (1 << i) / 2;
                    fft_bf(v[q], v[q + (1 << i)], w.im, -w.re);
                }
            }
        }
    }
#pragma unroll
    for (int a = 0; a < R; a++) v[a] = cpx_mul(v[a], turn[next + a].re, turn[next + a].im);
}

// ---- copies a thread block waits for, one after the other ----
//
// Every thread waits for the copy of a turn; one thread starts the next copy, behind a barrier of the block.  A thread has a
// number of tries for all its waits together, of which copies that come in time take none.  When they are used up it
// waits no more, and what it reads means nothing; if it is the one that starts the copies it starts no more, so
// that there are never two on their way, and it stays at the turn that it lost.
struct CopyTurns {
    uint32_t state;                                    // tries left, and the parity of the copy to come in bit 0
    explicit HD CopyTurns(uint32_t tries) : state(2 * tries) {}
    HD uint32_t parity() const { return state & 1u; }
    HD bool lost() const { return state < 2; }
    // try_once(parity): whether the copy is there, after a while
    template <class Try>
    HD bool take(const Try &try_once) {
        while (!lost()) {
            if (try_once(parity())) {
                state ^= 1u;
                return true;
            }
            state -= 2;
        }
        return false;
    }
};

#if defined(__CUDACC__)
// ---- whole blocks (device) -----------------------------------------------------------

// ---- barriers of a cluster ----
//
// The transform buffer is written after buffer_wait() and given free with buffer_free() after its last
// read, by whichever thread block of the cluster: the two halves of a barrier, with work in between.
// One free is open at the start of every step, and every block of a cluster takes the same steps.
__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire;" ::: "memory"); }
template <int CL>
__device__ __forceinline__ void buffer_wait() {
    if constexpr (CL > 0) cluster_wait();
    else __syncthreads();
}
template <int CL>
__device__ __forceinline__ void buffer_free() {
    if constexpr (CL > 0) cluster_arrive();
}
// x in layout A -> layout C (unscaled, with omega^-tid, without the registers' constants).  The
// buffer is not given free: its words in layout C are the thread's own.  has_read() runs when the thread has
// taken its values from there.
template <int CL, class Read>
__device__ __forceinline__ void fft_inverse(cpx (&x)[16], double2 *buf, const root_t *tab, uint32_t tid, const Read &has_read) {
    using L = FftLay;
    const uint32_t lane = tid & 31u;
    double2 *wb = buf + (tid >> 5) * 512;
    inv_phase_a(x);
    buffer_wait<CL>();
#pragma unroll
    for (int r = 0; r < 16; r++) wb[L::a_word(lane, r)] = make_double2(x[r].re, x[r].im);
    __syncwarp();
#pragma unroll
    for (int r = 0; r < 16; r++) {
        const double2 v = wb[L::b_word(lane, r)];
        x[r] = cpx{v.x, v.y};
    }
    inv_phase_b(x, tab, lane & 15u);
    __syncwarp();
#pragma unroll
    for (int r = 0; r < 16; r++) wb[L::bc_word(lane, r)] = make_double2(x[r].re, x[r].im);
    __syncthreads();
#pragma unroll
    for (int r = 0; r < 16; r++) {
        const double2 v = buf[tid + L::NT * r];
        x[r] = cpx{v.x, v.y};
    }
    has_read();
    inv_phase_c(x, tab + FftTab<0>::C, tid);
}

template <int CL>
__device__ __forceinline__ void fft_inverse(cpx (&x)[16], double2 *buf, const root_t *tab, uint32_t tid) {
    fft_inverse<CL>(x, buf, tab, tid, [] {});
}

// x in layout C -> layout A; block b of 2^CL blocks.  ALONE: outside a cluster.
template <int CL, bool ALONE = false>
__device__ __forceinline__ void fft_forward(cpx (&x)[16], double2 *buf, const root_t *fwd, uint32_t b, uint32_t tid) {
    using L = FftLay;
    const uint32_t lane = tid & 31u, warp = tid >> 5;
    double2 *wb = buf + warp * 512;
    const uint32_t top = (1u << CL) + b;                   // level CL, block b
    fwd_phase4_at(x, fwd, top);
    buffer_wait<ALONE ? 0 : CL>();
#pragma unroll
    for (int r = 0; r < 16; r++) buf[tid + L::NT * r] = make_double2(x[r].re, x[r].im);
    __syncthreads();
#pragma unroll
    for (int r = 0; r < 16; r++) {
        const double2 v = wb[L::bc_word(lane, r)];
        x[r] = cpx{v.x, v.y};
    }
    fwd_phase4_at(x, fwd, (top << 4) + 2 * warp + (lane >> 4));       // position bits 8 and up
    __syncwarp();
#pragma unroll
    for (int r = 0; r < 16; r++) wb[L::b_word(lane, r)] = make_double2(x[r].re, x[r].im);
    __syncwarp();
#pragma unroll
    for (int r = 0; r < 16; r++) {
        const double2 v = wb[L::a_word(lane, r)];
        x[r] = cpx{v.x, v.y};
    }
    buffer_free<ALONE ? 0 : CL>();
    fwd_phase4_last(x, fwd + (L::NB << CL) + b * FFT_LAST, tid);  // position bits 4 and up
}
#endif

}  // namespace fedhe

// Plays the complex transforms behind the exact products on the host, thread by thread, with the
// device's own index arithmetic, and compares products of a ternary polynomial and one of the largest
// pieces with the exact integers.  usage: host_fft_check logN, or 0 for the
// turns of a kernel's copies
#include <cstdio>
#include <cstdlib>
#include <random>
#include <vector>

#include "../include/fedhe.h"
#include "../paper_2303_10837_b200/csrc/fedhe_fft.cuh"
#include "../paper_2303_10837_b200/csrc/fedhe_host.h"

using namespace fedhe;

struct Block {
    using L = FftLay;
    std::vector<cpx> buf = std::vector<cpx>(L::NB);
    std::vector<std::vector<cpx>> reg = std::vector<std::vector<cpx>>(L::NT, std::vector<cpx>(16));

    template <class F>
    void each(F f) {
        for (uint32_t tid = 0; tid < (uint32_t)L::NT; tid++) {
            cpx x[16];
            for (int r = 0; r < 16; r++) x[r] = reg[tid][r];
            f(x, tid);
            for (int r = 0; r < 16; r++) reg[tid][r] = x[r];
        }
    }
    template <class W, class R>
    void exchange(W w, R r_) {
        std::vector<char> seen(L::NB, 0);
        for (uint32_t tid = 0; tid < (uint32_t)L::NT; tid++)
            for (int r = 0; r < 16; r++) {
                const uint32_t i = w(tid, r);
                if (i >= (uint32_t)L::NB || seen[i]++) { std::printf("a word is written twice\n"); std::exit(1); }
                buf[i] = reg[tid][r];
            }
        for (uint32_t tid = 0; tid < (uint32_t)L::NT; tid++)
            for (int r = 0; r < 16; r++) reg[tid][r] = buf[r_(tid, r)];
    }
    static uint32_t wa(uint32_t t, int r) { return (t >> 5) * 512 + L::a_word(t & 31u, r); }
    static uint32_t wb(uint32_t t, int r) { return (t >> 5) * 512 + L::b_word(t & 31u, r); }
    static uint32_t wbc(uint32_t t, int r) { return (t >> 5) * 512 + L::bc_word(t & 31u, r); }
    static uint32_t wc(uint32_t t, int r) { return t + L::NT * (uint32_t)r; }

    void forward(const root_t *fwd, uint32_t n, uint32_t top) {
        each([&](cpx (&x)[16], uint32_t) { fwd_phase4_at(x, fwd, top); });
        exchange(wc, wbc);
        each([&](cpx (&x)[16], uint32_t t) { fwd_phase4_at(x, fwd, (top << 4) + 2 * (t >> 5) + ((t & 31u) >> 4)); });
        exchange(wb, wa);
        const root_t *last = fwd + n + (top - n / L::NB) * FFT_LAST;
        each([&](cpx (&x)[16], uint32_t t) { fwd_phase4_last(x, last, t); });
    }
    void inverse(const root_t *tab) {
        each([&](cpx (&x)[16], uint32_t) { inv_phase_a(x); });
        exchange(wa, wb);
        each([&](cpx (&x)[16], uint32_t t) { inv_phase_b(x, tab, t & 15u); });
        exchange(wbc, wc);
        each([&](cpx (&x)[16], uint32_t t) { inv_phase_c(x, tab + FftTab<0>::C, t); });
    }
};

template <int CL>
static int check(uint32_t N) {
    using L = FftLay;
    constexpr uint32_t R = 1u << CL, NB = L::NB, NT = L::NT;
    const uint32_t n = N / 2;
    const int logN = 13 + CL;
    std::vector<double> roots, fwd, inv;
    std::vector<uint32_t> slot_of;
    host_unit_roots(N, roots);
    host_fft_tables(N, roots, fwd, inv, slot_of);
    if (inv.size() != 2 * (size_t)FftTab<CL>::WORDS) { std::printf("table size\n"); return 1; }
    const root_t *ft = reinterpret_cast<const root_t *>(fwd.data()), *it = reinterpret_cast<const root_t *>(inv.data());
    std::mt19937_64 rng(N);
    int bad = 0;
    for (int kind = 0; kind < 8; kind++) {
        // sure pieces: uniform, largest values with random signs, largest values of one sign; wide ones: uniform, of several
        // keys; and the low pieces of two limbs in one operand
        const bool wide = kind >= 3 && kind < 7, pair = kind == 7;
        const int low_bits = fft_random_bits(logN, 16, FFT_PAIR_EXPONENT);
        const int b = wide ? fft_wide_bits(logN) : pair ? 16 + low_bits : fft_sure_bits(logN);
        const double sd = fft_error_sd(logN, b);
        // of 2^16 errors the largest is near 4.3 standard deviations, and 8 are never seen
        const double bound = wide || pair ? 8 * sd : (11.4 * (logN - 1) + 23.0) * std::ldexp(1.0, logN + b - 1 - 53);
        std::vector<int64_t> p(N), u(N), low[2] = {std::vector<int64_t>(N), std::vector<int64_t>(N)};
        const int64_t top = (int64_t)1 << (b - 1);
        for (uint32_t i = 0; i < N; i++) {
            low[0][i] = (int64_t)(rng() >> (64 - low_bits)) - ((int64_t)1 << (low_bits - 1));
            low[1][i] = (int64_t)(rng() >> (64 - low_bits)) - ((int64_t)1 << (low_bits - 1));
            p[i] = pair ? low[0][i] + 65536 * low[1][i] : kind == 0 || wide ? (int64_t)(rng() >> (64 - b)) - top : kind == 1 ? ((rng() & 1) ? top : -top) : top;
            u[i] = kind == 2 ? 1 : (int64_t)(rng() % 3) - 1;
        }
        auto transform = [&](const std::vector<int64_t> &a, uint32_t blk, Block &B) {
            const OuterPath<CL> outer(ft, blk);
            B.each([&](cpx (&x)[16], uint32_t tid) {
                for (int r = 0; r < 16; r++) {
                    cpx z[R], y[R];
                    for (uint32_t w = 0; w < R; w++) {
                        const uint32_t k = w * NB + tid + NT * r;
                        y[w] = z[w] = cpx{(double)a[k], (double)a[k + n]};
                    }
                    x[r] = outer.apply(z);
                    fft_outer_forward<CL>(y, ft);       // all blocks at once: the same value
                    if (std::fabs(y[blk].re - x[r].re) + std::fabs(y[blk].im - x[r].im) > 1e-15 * 4 * R * (double)top) {
                        std::printf("outer stages\n");
                        std::exit(1);
                    }
                }
            });
            B.forward(ft, n, R + blk);
        };
        std::vector<Block> prod(R);
        for (uint32_t blk = 0; blk < R; blk++) {
            Block bu;
            transform(p, blk, prod[blk]);
            transform(u, blk, bu);
            if (kind == 0 && blk == R - 1) {     // a slot's value, straight from the definition
                const uint32_t tid = NT / 3, r = 5, j = slot_of[(blk * 16 + r) * NT + tid];
                uint64_t e = 1;
                for (uint32_t k = 0; k < j; k++) e = e * 5 % (2 * N);
                long double v = 0;
                for (uint32_t k = 0; k < N; k++) v += (long double)u[k] * roots[2 * (size_t)((e * k) % (2 * N))];
                if (std::fabs((double)(v - bu.reg[tid][r].re)) > 1e-9) { std::printf("slot order\n"); bad = 1; }
            }
            for (uint32_t w = 0; w < NB; w++)    // the slots of a block have one residue mod R
                if (slot_of[blk * NB + w] % R != slot_of[blk * NB] % R) { std::printf("slot residue\n"); return 1; }
            prod[blk].each([&](cpx (&x)[16], uint32_t tid) {
                for (int r = 0; r < 16; r++) {
                    x[r] = cpx_mul(x[r], bu.reg[tid][r].re, bu.reg[tid][r].im);
                    x[r].re /= n;
                    x[r].im /= n;
                }
            });
            prod[blk].inverse(it);
        }
        std::vector<double> c(N);
        for (uint32_t tid = 0; tid < NT; tid++)
            for (uint32_t r = 0; r < 16; r++) {
                cpx v[R];
                for (uint32_t w = 0; w < R; w++) v[w] = prod[w].reg[tid][r];
                fft_outer_inverse<CL>(v, it, tid, r);
                for (uint32_t w = 0; w < R; w++) {
                    c[w * NB + tid + NT * r] = v[w].re;
                    c[w * NB + tid + NT * r + n] = v[w].im;
                }
            }
        double worst = 0;
        for (int s = 0; s < 300; s++) {           // single coefficients against the schoolbook sum
            const uint32_t k = s < 4 ? (s & 1 ? N - 1 - s / 2 : s / 2) : (uint32_t)(rng() % N);
            auto product = [&](const std::vector<int64_t> &a) {
                int64_t sum = 0;
                for (uint32_t i = 0; i < N; i++) sum += i <= k ? u[i] * a[k - i] : -u[i] * a[N + k - i];
                return sum;
            };
            const int64_t want = product(p);
            if (pair) {                           // each limb's product out of the rounded word
                const int64_t z = (int64_t)std::nearbyint(c[k]), first = (int16_t)z;
                if (first != product(low[0]) || (z - first) >> 16 != product(low[1])) { std::printf("pair of limbs\n"); bad = 1; }
            }
            worst = std::max(worst, std::fabs(c[k] - (double)want));
        }
        double off = 0, sq = 0;                   // and the distance of all of them to an integer
        for (uint32_t k = 0; k < N; k++) {
            const double d = std::fabs(c[k] - std::nearbyint(c[k]));
            off = std::max(off, d);
            sq += d * d;
        }
        std::printf("N %u, %d bits, kind %d: error %.3g, off an integer %.3g (rms %.3g, model %.3g), bound %.3g\n", N, b, kind, worst,
                    off, std::sqrt(sq / N), sd, bound);
        if (!(worst < bound) || !(off < bound)) bad = 1;
        if (wide && std::sqrt(sq / N) > sd) bad = 1;
    }
    return bad;
}

// A thread block whose threads, in any order, wait for copies of which one comes late or never: there are never two on
// their way, none is started after the starting thread lost one, and every wait ends.
static void copies_that_do_not_come() {
    std::mt19937 rng(7);
    const int NT = 8, TURNS = 8;
    const uint32_t TRIES = 6;
    for (int trial = 0; trial < 20000; trial++) {
        const int bad = (int)(rng() % (TURNS + 1));          // TURNS: every copy comes in time
        const bool never = rng() % 2;
        struct Thread { CopyTurns turns{TRIES}; int turn = 0; uint32_t tries = 0; bool behind = false; } th[NT];
        int arrived[TURNS] = {}, started = 1, phases = 0, running = NT;      // phases of the copies' barrier that are over
        while (running) {
            const int id = (int)(rng() % NT);
            Thread &t = th[id];
            if (t.turn == TURNS) continue;
            if (!t.behind) {
                // a try goes on for longer than a copy that comes in time takes, and than the others' way to the barrier
                if (started <= t.turn && !th[0].turns.lost() && !t.turns.lost()) continue;
                t.turns.take([&](uint32_t parity) {
                    if (phases < started && (phases != bad || (!never && rng() % 16 == 0))) phases++;
                    const bool here = (uint32_t)(phases & 1) != parity;
                    t.tries += !here;
                    return here;
                });
                arrived[t.turn]++;
                t.behind = true;
            } else if (arrived[t.turn] == NT) {
                if (id == 0 && t.turn + 1 < TURNS && !t.turns.lost()) {
                    if (phases != started) { std::printf("two copies at once\n"); std::exit(1); }
                    started++;
                }
                t.behind = false;
                running -= ++t.turn == TURNS;
            }
        }
        bool lost = false;
        for (const Thread &t : th) {
            lost = lost || t.turns.lost();
            if (t.tries > TRIES) { std::printf("the waits are too long\n"); std::exit(1); }
        }
        if ((lost && bad == TURNS) || (!th[0].turns.lost() && started != TURNS) ||
            (th[0].turns.lost() && (started != bad + 1 || th[0].turns.parity() != (uint32_t)(bad & 1)))) {
            std::printf("a lost copy is not the last\n");
            std::exit(1);
        }
    }
    if (host_status_code(0) != HE_OK || host_status_code(STATUS_RANGE) != HE_ERR_OVERFLOW || host_status_code(STATUS_COPY) != HE_ERR_CUDA ||
        host_status_code(STATUS_RANGE | STATUS_COPY) != HE_ERR_CUDA) {
        std::printf("status codes\n");
        std::exit(1);
    }
}

int main(int argc, char **argv) {
    const int logN = argc > 1 ? std::atoi(argv[1]) : 13;
    int bad = 0;
    if (logN == 0) copies_that_do_not_come();
    if (logN == 13) bad |= check<0>(1u << 13);
    if (logN == 14) bad |= check<1>(1u << 14);
    if (logN == 15) bad |= check<2>(1u << 15);
    if (logN == 16) bad |= check<3>(1u << 16);
    std::puts(bad ? "FAILED" : "ok");
    return bad;
}

// Mask selection, packing and merging kernels (part 6 of the kernels).
#include "fedhe_kernels.cuh"

namespace fedhe {

// ===========================================================================
// selective-encryption mask
// ===========================================================================

// ordering key of a sensitivity score: its bit pattern when it is a
// non-negative number, 0 for negatives, -0 and NaN
__device__ __forceinline__ uint32_t score_key(float s) {
    const uint32_t b = __float_as_uint(s);
    return b > 0x7f800000u ? 0u : b;                       // the sign bit is above all of these
}

// exclusive prefix sum over the threads of a block (any whole number of warps up to 32); the block total goes to `total`
template <class T>
__device__ __forceinline__ T block_exclusive_scan(T v, T *warp_sums, T &total) {
    const uint32_t lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    T inc = v;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const T o = __shfl_up_sync(0xffffffffu, inc, d);
        if (lane >= (uint32_t)d) inc += o;
    }
    if (lane == 31) warp_sums[warp] = inc;
    __syncthreads();
    if (warp == 0) {
        T w = lane < ((blockDim.x + 31u) >> 5) ? warp_sums[lane] : (T)0, winc = w;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const T o = __shfl_up_sync(0xffffffffu, winc, d);
            if (lane >= (uint32_t)d) winc += o;
        }
        warp_sums[lane] = winc - w;          // exclusive warp offsets
        if (lane == 31) warp_sums[32] = winc;
    }
    __syncthreads();
    const T res = warp_sums[warp] + inc - v;
    total = warp_sums[32];
    __syncthreads();
    return res;
}

// ---- selection of the k-th largest key ----
//
// A window of keys that holds the threshold, 2^20 to 2^22 of them by a sample of the scores or 2^20 by the histogram of the keys' first
// digit (11 of their 31 bits); one pass over the scores that counts and marks the keys beyond the window and
// gathers those within (the candidates, a few per cent of real scores) by tiles; then a digit of ten bits, one of the 10 to 12 that are left
// and the marking on the candidates.  The last thread block of a pass to finish does the one-block step that follows it: picking the digit, or
// the scan over the tiles.  For 2.56 M out of 25.6 M scores the call took 341 us by three histogram passes, a counting pass
// and one-block kernels between them (conflicts of shared-memory atomics, because neighbouring scores share an exponent), 165 us
// with the histogram of the first digit over all scores (27 us) and the scores read again for the marking (33 us).

// true in all threads of the block that finishes last; what the others wrote is visible to it
__device__ __forceinline__ bool last_block(uint32_t *done) {
    __shared__ uint32_t is_last;
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) is_last = atomicAdd(done, 1u) + 1u == gridDim.x ? 1u : 0u;
    __syncthreads();
    if (is_last) __threadfence();
    return is_last != 0;
}

// Calls see(digit, keys above it, its keys) for every digit of a histogram, by one thread each.  By a block of NT threads.
template <int BITS, uint32_t NT = 1024, class See>
__device__ __forceinline__ void radix_walk(const uint32_t *hist, const See &see) {
    __shared__ uint32_t warp_sums[33];
    constexpr uint32_t bins = 1u << BITS, per = bins / NT;           // thread t: digits from bins - 1 - per t down
    uint32_t h[per], mine = 0u;
#pragma unroll
    for (uint32_t j = 0; j < per; j++) {
        h[j] = __ldcg(hist + bins - 1u - (threadIdx.x * per + j));
        mine += h[j];
    }
    uint32_t tot;
    uint32_t above = block_exclusive_scan(mine, warp_sums, tot);     // keys in digits above this thread's
#pragma unroll
    for (uint32_t j = 0; j < per; j++) {
        const uint32_t pos = threadIdx.x * per + j;
        see(bins - 1u - pos, above, h[j]);
        above += h[j];
    }
}
// found(digit, keys above it) for the digit where the count from the largest down first reaches `need`, if there are as many
template <int BITS, uint32_t NT = 1024, class Found>
__device__ __forceinline__ void radix_pick(const uint32_t *hist, uint32_t need, const Found &found) {
    radix_walk<BITS, NT>(hist, [&](uint32_t digit, uint32_t above, uint32_t count) {
        if (above < need && above + count >= need) found(digit, above);
    });
}

// First digit.  Every lane counts in a column of its own, so the lanes of a warp never meet in a word or a bank: two
// 16-bit counters to a word, [1024][32].  A column takes a 32nd of the block's keys, and a block at most HIST_KEYS.
constexpr int LOADS = 8, HIST_LOADS = 16;
constexpr size_t HIST_KEYS = 32 * 65536 - 2048, HIST_SMEM = 1024 * 32 * sizeof(uint32_t);

__global__ void __launch_bounds__(1024, 1)
key_histogram_kernel(const float *score, size_t P, SelectWork w, uint32_t k) {
    extern __shared__ uint32_t sh[];
    const uint32_t lane = threadIdx.x & 31u;
    for (uint32_t b = threadIdx.x; b < 1024u * 32u; b += 1024u) sh[b] = 0;
    __syncthreads();
    uint32_t *mine = sh + lane;
    const size_t step = (size_t)gridDim.x * 1024u;
    auto count = [&](float v) {
        const uint32_t d = score_key(v) >> 20;
        atomicAdd(mine + (d >> 1) * 32u, 1u << ((d & 1u) * 16u));
    };
    size_t i = (size_t)blockIdx.x * 1024u + threadIdx.x;
    if (i + (HIST_LOADS - 1) * step < P) {
        // the next loads are on their way while these are counted
        float v[HIST_LOADS];
#pragma unroll
        for (int j = 0; j < HIST_LOADS; j++) v[j] = __ldg(score + i + j * step);
        for (i += step * HIST_LOADS; i + (HIST_LOADS - 1) * step < P; i += step * HIST_LOADS) {
            float next[HIST_LOADS];
#pragma unroll
            for (int j = 0; j < HIST_LOADS; j++) next[j] = __ldg(score + i + j * step);
#pragma unroll
            for (int j = 0; j < HIST_LOADS; j++) count(v[j]);
#pragma unroll
            for (int j = 0; j < HIST_LOADS; j++) v[j] = next[j];
        }
#pragma unroll
        for (int j = 0; j < HIST_LOADS; j++) count(v[j]);
    }
    for (; i < P; i += 4 * step) {
        float v[4];
#pragma unroll
        for (int j = 0; j < 4; j++) v[j] = i + j * step < P ? __ldg(score + i + j * step) : 0.0f;
#pragma unroll
        for (int j = 0; j < 4; j++)
            if (i + j * step < P) count(v[j]);
    }
    __syncthreads();
    uint32_t even = 0, odd = 0;
#pragma unroll
    for (uint32_t j = 0; j < 32u; j++) {
        const uint32_t c = sh[threadIdx.x * 32u + ((lane + j) & 31u)];
        even += c & 0xffffu;
        odd += c >> 16;
    }
    if (even) atomicAdd(w.hist + 2 * threadIdx.x, even);
    if (odd) atomicAdd(w.hist + 2 * threadIdx.x + 1, odd);
    if (last_block(w.done)) {
        if (k == 0) {
            if (threadIdx.x == 0) w.state->base = 0x80000000u;                   // no key reaches the window
        } else {
            radix_pick<11>(w.hist, k, [&](uint32_t digit, uint32_t) { w.state->base = digit << 20; });
        }
    }
}

// The window from a sample: a score at a pseudo-random place of every SAMPLE-th part of them, in a histogram of the keys'
// upper 12 bits of 31.  The threshold is surely between the bins of two places in the sample (SampleRanks); the last block puts a window of 2^20,
// 2^21 or 2^22 keys around these, or leaves it to the histogram of all keys.  A block counts in shared memory: sampled keys share some
// hundred bins, and as atomics in L2 they took 58 us.
constexpr uint32_t SAMPLE_BLOCKS = 128, SAMPLE_LOADS = 2, SAMPLE = SAMPLE_BLOCKS * SAMPLE_LOADS * 1024;
static_assert(SELECT_BINS == 1u << 12, "bins of 2^19 keys");
struct SampleRanks { uint32_t first, last; };

__global__ void __launch_bounds__(1024, 1) key_sample_kernel(const float *score, size_t P, SelectWork w, SampleRanks r) {
    __shared__ __align__(16) uint32_t sh[SELECT_BINS];
    __shared__ uint32_t upper, lower;
    const size_t step = P / SAMPLE;
    float v[SAMPLE_LOADS];
#pragma unroll
    for (uint32_t j = 0; j < SAMPLE_LOADS; j++) {
        const uint32_t i = (blockIdx.x * SAMPLE_LOADS + j) * 1024u + threadIdx.x;
        v[j] = __ldg(score + i * step + (uint32_t)(((uint64_t)(i * 2654435761u) * step) >> 32));
    }
    for (uint32_t b = threadIdx.x; b < SELECT_BINS / 4; b += 1024u) reinterpret_cast<uint4 *>(sh)[b] = make_uint4(0, 0, 0, 0);
    __syncthreads();
#pragma unroll
    for (uint32_t j = 0; j < SAMPLE_LOADS; j++) atomicAdd(sh + (score_key(v[j]) >> 19), 1u);
    __syncthreads();
    for (uint32_t b = threadIdx.x; b < SELECT_BINS; b += 1024u)
        if (sh[b]) atomicAdd(w.sampled + b, sh[b]);
    if (!last_block(w.done + 4)) return;
    radix_walk<12>(w.sampled, [&](uint32_t bin, uint32_t above, uint32_t count) {
        if (above < r.first && above + count >= r.first) upper = bin;
        if (above < r.last && above + count >= r.last) lower = bin;
    });
    __syncthreads();
    if (threadIdx.x) return;
    const uint32_t bins = upper - lower + 1u, shift = bins <= 2u ? 0u : bins <= 4u ? 1u : bins <= 8u ? 2u : WINDOW_OPEN;
    w.state->shift = shift;
    if (shift == WINDOW_OPEN) return;
    const uint32_t under = ((2u << shift) - bins) << 18, from = lower << 19;       // what is left over goes to both sides
    w.state->base = from > under ? from - under : 0u;
}

// The standard deviation of a sample's share of k is sqrt(p (1 - p) / SAMPLE): 0.6, 1.9 and 3.1 % of p = 0.1, 0.01 and 1 / 256.  Four of them to either
// side move the threshold by 2, 3 and 5 % for scores that are products of two normal variables, and by 12 % for log-normal ones whose logarithm
// has a standard deviation of 3 and p = 0.005; the windows are at least 6, 12 and 25 % wide.  Scores in a wider spread go by the histogram
// (155 us; 140 without the sample).  With one window of 2^20 keys around the place that 131,072 samples guessed, log-normal scores missed it in up to
// half of all selections, and a miss costs the whole selection again (25.6 M scores, 1 in 200 of them: 181 us instead of 100).  Fewer scores beyond the
// threshold, or in all, go by the histogram of all: at 2.5 M scores that is as quick (88 us and 90).
bool select_by_sample(size_t P, size_t k) { return P >= (size_t)1 << 22 && k >= P / 256 && P - k >= P / 256; }
static SampleRanks sample_ranks(size_t P, size_t k) {
    const double p = (double)k / (double)P, mean = p * SAMPLE, off = 4.0 * sqrt(mean * (1.0 - p));
    return SampleRanks{(uint32_t)(mean - off), (uint32_t)(mean + off) + 2u};         // within 1 .. SAMPLE: k and P - k are P / 256 at least
}

// f(first word, words' keys) for LOADS words of a tile at a time, by a warp: lane l the l-th parameter of each word.
// Beyond the end keys are 0, and f is told how many parameters are left (LOADS * 32 or less).
template <class F>
__device__ __forceinline__ void for_tile(const float *score, size_t P, size_t first, F f) {
    const uint32_t lane = threadIdx.x & 31u;
    const float *p = score + first + lane;
    const uint32_t left = P - first < MASK_BLOCK ? (uint32_t)(P - first) : MASK_BLOCK;
#pragma unroll 1
    for (uint32_t w0 = 0; w0 * 32 < left; w0 += LOADS) {
        uint32_t key[LOADS];
        if ((w0 + LOADS) * 32 <= left) {
#pragma unroll
            for (int j = 0; j < LOADS; j++) key[j] = score_key(__ldg(p + (w0 + j) * 32));
            f(w0, key, LOADS * 32u);
        } else {
#pragma unroll
            for (int j = 0; j < LOADS; j++)
                key[j] = (w0 + j) * 32 + lane < left ? score_key(__ldg(p + (w0 + j) * 32)) : 0u;
            f(w0, key, left - w0 * 32);
        }
    }
}

// The pass over the scores.  A warp takes a tile of MASK_BLOCK of them, marks and counts the keys beyond the window and gathers those
// within, lane by lane: the place in the tile and the key less the window's base, 22 bits.  A tile with more than TILE_CANDIDATES of
// them is read again instead.  It is bound by its instructions, so the scores' bit patterns themselves are compared (a key is 0 where
// they are not those of a number from 0 to infinity, and only a window at 0 holds such keys), and a lane only notes its candidates in a word,
// and reads them again at the tile's end (gathering them word by word took 52 us for 25.6 M scores).
__device__ __forceinline__ uint32_t window_place(uint32_t key, uint32_t base) { return key - base; }        // below the number of its keys within
constexpr int CAND_THREADS = 512;
__global__ void __launch_bounds__(CAND_THREADS, 3)
key_candidates_kernel(const float *score, size_t P, SelectWork w, uint32_t k) {
    __shared__ uint32_t sh[1024], beyond;
    if (w.state->shift == WINDOW_OPEN) {
        if (blockIdx.x == 0 && threadIdx.x == 0) w.total[1] = 1u;
        return;
    }
    for (uint32_t b = threadIdx.x; b < 1024u; b += CAND_THREADS) sh[b] = 0;
    if (threadIdx.x == 0) beyond = 0;
    __syncthreads();
    const uint32_t base = w.state->base, shift = w.state->shift, keys = 1u << (20 + shift), infinity = 0x7f800000u;
    // bit patterns beyond the window and within: from `last` + 1 and from `base`, so many
    const uint32_t last = base + keys - 1u, many = infinity > last ? infinity - last : 0u;
    const uint32_t within = base > infinity ? 0u : infinity - base < keys - 1u ? infinity - base + 1u : keys;
    // in a window at 0, where a key of 0 has many bit patterns, is all that is not beyond it
    const uint32_t in_from = base ? base : last + 1u, in_many = base ? within : many, turned = base ? 0u : 0xffffffffu;
    const uint32_t lane = threadIdx.x & 31u;
    const size_t tiles = (P + MASK_BLOCK - 1) / MASK_BLOCK, whole = P / MASK_BLOCK, stride = (size_t)gridDim.x * (CAND_THREADS / 32);
    size_t tile = (size_t)blockIdx.x * (CAND_THREADS / 32) + (threadIdx.x >> 5);
    uint32_t all_above = 0;
    const float *p = score + tile * MASK_BLOCK + lane;
    // the next words are on their way while these are looked at
    float next[LOADS];
    if (tile < whole) {
#pragma unroll
        for (int j = 0; j < LOADS; j++) next[j] = __ldg(p + j * 32);
    }
#pragma unroll 1
    for (; tile < tiles; tile += stride, p += stride * MASK_BLOCK) {
        uint32_t my_bits = 0, mine = 0;                             // word `lane` of the marks; bit i: the lane's key in word i is a candidate
        static_assert(MASK_BLOCK == 1024, "a word of the tile for every lane");
        if (tile < whole) {
#pragma unroll 1
            for (uint32_t w0 = 0; w0 < 32; w0 += LOADS) {
                uint32_t who[LOADS], some = 0;
#pragma unroll
                for (int j = 0; j < LOADS; j++) {
                    const uint32_t raw = __float_as_uint(next[j]);
                    who[j] = __ballot_sync(0xffffffffu, raw - last - 1u < many);
                    if (raw - in_from < in_many) some |= 1u << j;
                }
                mine |= some << w0;
                const bool same = w0 + LOADS < 32;
                const float *q = same ? p + (w0 + LOADS) * 32 : p + stride * MASK_BLOCK;
                if (same || tile + stride < whole) {
#pragma unroll
                    for (int j = 0; j < LOADS; j++) next[j] = __ldg(q + j * 32);
                }
                // the word of the lane's number among these
                static_assert(LOADS == 8, "three bits pick it");
                const uint32_t a = lane & 1u ? who[1] : who[0], b = lane & 1u ? who[3] : who[2], c = lane & 1u ? who[5] : who[4],
                               d = lane & 1u ? who[7] : who[6], e = lane & 2u ? b : a, f = lane & 2u ? d : c;
                if ((lane & ~7u) == w0) my_bits = lane & 4u ? f : e;
            }
            mine ^= turned;
        } else {
            const uint32_t left = (uint32_t)(P - tile * MASK_BLOCK);        // the last tile
#pragma unroll 1
            for (uint32_t word = 0; word < 32; word++) {
                const bool there = word * 32 + lane < left;
                const uint32_t key = there ? score_key(__ldg(p + word * 32)) : 0u;
                const uint32_t who = __ballot_sync(0xffffffffu, key > last);
                if (lane == word) my_bits = who;
                if (there && window_place(key, base) < keys) mine |= 1u << word;
            }
        }
        uint32_t at = __popc(mine);
        const uint32_t n = at;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const uint32_t o = __shfl_up_sync(0xffffffffu, at, d);
            if (lane >= (uint32_t)d) at += o;
        }
        const uint32_t found = __shfl_sync(0xffffffffu, at, 31);
        at -= n;
        uint32_t *cand = w.cand + tile * TILE_CANDIDATES;
        while (mine) {
            constexpr int A = 4;
            uint32_t word[A];
            float v[A];
#pragma unroll
            for (int i = 0; i < A; i++) {
                word[i] = mine ? __ffs((int)mine) - 1 : 32;
                mine &= mine - 1u;                                  // 0 stays 0
                v[i] = word[i] < 32 ? __ldg(p + word[i] * 32) : 0.0f;
            }
#pragma unroll
            for (int i = 0; i < A; i++) {
                if (word[i] == 32) break;
                const uint32_t low = window_place(score_key(v[i]), base);
                if (at < TILE_CANDIDATES) cand[at] = low << 10 | (word[i] * 32u + lane);
                at++;
                atomicAdd(sh + (low >> (10 + shift) & 1023u), 1u);
            }
        }
        if (tile < whole || lane * 32u < P - tile * MASK_BLOCK) w.bits[tile * (MASK_BLOCK / 32) + lane] = my_bits;
        const uint32_t above = __reduce_add_sync(0xffffffffu, __popc(my_bits));
        all_above += above;
        if (lane == 0) {
            w.tile_above[tile] = above;
            w.tile_cand[tile] = found;
            w.tile_found[tile] = found;
        }
    }
    if (lane == 0 && all_above) atomicAdd(&beyond, all_above);
    __syncthreads();
    for (uint32_t b = threadIdx.x; b < 1024u; b += CAND_THREADS)
        if (sh[b]) atomicAdd(w.hist + 2048 + b, sh[b]);
    if (threadIdx.x == 0 && beyond) atomicAdd(&w.state->above, beyond);
    if (!last_block(w.done + 1)) return;
    const uint32_t too_many = __ldcg(&w.state->above);
    if (threadIdx.x == 0) w.total[1] = k ? 1u : 0u;                    // until the threshold is found
    __syncthreads();
    if (k > too_many)
        radix_pick<10, CAND_THREADS>(w.hist + 2048, k - too_many, [&](uint32_t digit, uint32_t over) {
            w.state->place = digit;
            w.state->need = k - too_many - over;
            w.total[1] = 0u;
        });
}

// f(in, place in the window and, below it, in the tile) for the listed candidates of a tile, by a whole warp: the lane's every 32nd, of which the
// first is there already (rarely more than 32: these come with their number)
template <class F>
__device__ __forceinline__ void for_listed(const uint32_t *cand, uint32_t c, uint32_t found, F f) {
    const uint32_t lane = threadIdx.x & 31u;
    for (uint32_t i = 0; i < found; i += 32) {
        const bool in = i + lane < found;
        f(in, in ? c : 0u);
        if (i + 32 < found) c = cand[i + 32];
    }
}

// the same for all candidates, of which there may be too many for the list
template <class F>
__device__ __forceinline__ void for_candidates(const float *score, size_t P, const SelectWork &w, size_t tile, uint32_t base, uint32_t keys, F f) {
    const uint32_t lane = threadIdx.x & 31u, found = w.tile_found[tile];
    const uint32_t *cand = w.cand + tile * TILE_CANDIDATES + lane;
    const uint32_t c0 = *cand;
    if (found <= TILE_CANDIDATES) {
        for_listed(cand, c0, found, f);
    } else {
        for_tile(score, P, tile * MASK_BLOCK, [&](uint32_t w0, const uint32_t (&key)[LOADS], uint32_t left) {
#pragma unroll
            for (int j = 0; j < LOADS; j++) {
                const uint32_t low = window_place(key[j], base);
                f(j * 32u + lane < left && low < keys, low << 10 | ((w0 + j) * 32u + lane));
            }
        });
    }
}

// the second digit, of the 10 to 12 bits that are left, over the candidates
__global__ void __launch_bounds__(1024, 2) key_last_digit_kernel(const float *score, size_t P, SelectWork w) {
    __shared__ uint32_t sh[SELECT_LAST];
    if (w.total[1]) return;                               // not in the window
    const uint32_t base = w.state->base, shift = w.state->shift, digit = w.state->place, need = w.state->need, digits = 1024u << shift;
    for (uint32_t b = threadIdx.x; b < digits; b += 1024u) sh[b] = 0;
    __syncthreads();
    const size_t tiles = (P + MASK_BLOCK - 1) / MASK_BLOCK;
    for (size_t tile = (size_t)blockIdx.x * 32u + (threadIdx.x >> 5); tile < tiles; tile += (size_t)gridDim.x * 32u)
        for_candidates(score, P, w, tile, base, 1u << (20 + shift), [&](bool in, uint32_t c) {
            if (in && c >> (20 + shift) == digit) atomicAdd(sh + (c >> 10 & (digits - 1u)), 1u);
        });
    __syncthreads();
    for (uint32_t b = threadIdx.x; b < digits; b += 1024u)
        if (sh[b]) atomicAdd(w.hist + 3072 + b, sh[b]);
    if (last_block(w.done + 2) && need)
        radix_pick<12>(w.hist + 3072, need, [&](uint32_t low, uint32_t over) {
            w.state->place = digit << (10 + shift) | low;
            w.state->need = need - over;
        });
}

// Keys above and equal to tau: a block takes a run of tiles, and leaves for each the counts before it within the run
// (equal keys in the upper half); the last block does the same for the runs.
__global__ void __launch_bounds__(1024, 2) tile_counts_kernel(const float *score, size_t P, SelectWork w) {
    __shared__ uint64_t warp_sums[33];
    if (w.total[1]) return;                               // not in the window
    const uint32_t base = w.state->base, keys = 1u << (20 + w.state->shift), place = w.state->place, need = w.state->need, lane = threadIdx.x & 31u;
    const size_t tiles = (P + MASK_BLOCK - 1) / MASK_BLOCK;
    const size_t begin = (size_t)blockIdx.x * w.run, end = begin + w.run < tiles ? begin + w.run : tiles;
    for (size_t tile = begin + (threadIdx.x >> 5); tile < end; tile += 32u) {
        uint32_t gt = 0, eq = 0;
        for_candidates(score, P, w, tile, base, keys, [&](bool in, uint32_t c) {
            gt += in && c >> 10 > place ? 1u : 0u;
            eq += in && c >> 10 == place ? 1u : 0u;
        });
        gt = __reduce_add_sync(0xffffffffu, gt);
        eq = __reduce_add_sync(0xffffffffu, eq);
        if (lane == 0) {
            w.tile_above[tile] += gt;
            w.tile_cand[tile] = eq;
        }
    }
    __syncthreads();
    uint64_t before = 0, tot;
    for (size_t t0 = begin; t0 < end; t0 += 1024u) {
        const size_t tile = t0 + threadIdx.x;
        const uint64_t c = tile < end ? ((uint64_t)w.tile_cand[tile] << 32) | w.tile_above[tile] : 0u;
        const uint64_t at = before + block_exclusive_scan(c, warp_sums, tot);
        before += tot;
        if (tile < end) {
            w.tile_cand[tile] = (uint32_t)(at >> 32);
            w.tile_above[tile] = (uint32_t)at;
        }
    }
    if (threadIdx.x == 0) __stcg(reinterpret_cast<unsigned long long *>(w.runs + blockIdx.x), (unsigned long long)before);
    if (!last_block(w.done + 3)) return;
    before = 0;
    for (uint32_t r0 = 0; r0 < gridDim.x; r0 += 1024u) {
        const uint32_t r = r0 + threadIdx.x;
        const uint64_t c = r < gridDim.x ? __ldcg(reinterpret_cast<const unsigned long long *>(w.runs + r)) : 0u;
        const uint64_t at = before + block_exclusive_scan(c, warp_sums, tot);
        before += tot;
        if (r < gridDim.x) w.runs[r] = at;
    }
    const uint32_t eq_all = (uint32_t)(before >> 32);
    if (threadIdx.x == 0) *w.total = (uint32_t)before + (eq_all < need ? eq_all : need);
}

cudaError_t launch_select(const float *score, size_t P, size_t k, bool by_sample, SelectWork &w, int n_sm, cudaStream_t s) {
    cudaError_t e;
    if ((e = cudaMemsetAsync(w.hist, 0, (SELECT_ZEROED + (by_sample ? SELECT_BINS : 0)) * sizeof(uint32_t), s))) return e;
    if (by_sample) {
        key_sample_kernel<<<SAMPLE_BLOCKS, 1024, 0, s>>>(score, P, w, sample_ranks(P, k));
        if ((e = FEDHE_LAUNCHED())) return e;
    }
    if ((e = cudaFuncSetAttribute(key_histogram_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)HIST_SMEM))) return e;
    // One thread block of the first pass to an SM, unless its counters could overflow; two keys to a thread are enough (with
    // sixteen, 100 k scores left a thread fourteen loads one after the other: 10 us more).
    const unsigned want = blocks_for(P, 1024 * 2), least = blocks_for(P, (unsigned)HIST_KEYS);
    unsigned g1 = want < (unsigned)n_sm ? want : (unsigned)n_sm;
    if (g1 < least) g1 = least;
    if (!by_sample) {
        key_histogram_kernel<<<g1, 1024, HIST_SMEM, s>>>(score, P, w, (uint32_t)k);
        if ((e = FEDHE_LAUNCHED())) return e;
    }
    auto grid = [&](unsigned per_block) {
        const unsigned blocks = blocks_for(P, per_block), resident = n_sm < 1024 ? 2u * (unsigned)n_sm : (unsigned)SELECT_RUNS;
        return blocks < resident ? blocks : resident;
    };
    const unsigned cand_blocks = blocks_for(P, CAND_THREADS / 32 * MASK_BLOCK), cand_fit = 3u * (unsigned)n_sm;
    key_candidates_kernel<<<cand_blocks < cand_fit ? cand_blocks : cand_fit, CAND_THREADS, 0, s>>>(score, P, w, (uint32_t)k);
    if ((e = FEDHE_LAUNCHED())) return e;
    key_last_digit_kernel<<<grid(32 * MASK_BLOCK), 1024, 0, s>>>(score, P, w);
    if ((e = FEDHE_LAUNCHED())) return e;
    const size_t tiles = (P + MASK_BLOCK - 1) / MASK_BLOCK;
    w.run = (uint32_t)((tiles + grid(32 * MASK_BLOCK) - 1) / grid(32 * MASK_BLOCK));
    tile_counts_kernel<<<(unsigned)((tiles + w.run - 1) / w.run), 1024, 0, s>>>(score, P, w);
    return FEDHE_LAUNCHED();
}

// single-block exclusive scan of an array (block totals: about a hundred
// thousand entries for the largest model): every thread sums a contiguous
// chunk, the chunk sums are scanned across the block, and the thread writes
// the running prefix back over its chunk
__global__ void __launch_bounds__(1024) scan_kernel(uint32_t *a, size_t count, uint32_t *total_out) {
    __shared__ uint32_t warp_sums[33];
    const size_t per = (count + 1023) / 1024;
    const size_t b = threadIdx.x * per, e = b + per < count ? b + per : count;
    uint32_t sum = 0;
    for (size_t i = b; i < e; i++) sum += a[i];
    uint32_t tot;
    uint32_t run = block_exclusive_scan(sum, warp_sums, tot);
    for (size_t i = b; i < e; i++) {
        const uint32_t v = a[i];
        a[i] = run;
        run += v;
    }
    if (threadIdx.x == 0) *total_out = tot;
}

cudaError_t launch_scan(uint32_t *a, size_t count, uint32_t *total, cudaStream_t s) {
    scan_kernel<<<1, 1024, 0, s>>>(a, count, total);
    return FEDHE_LAUNCHED();
}

// Membership: key > tau, or key == tau and fewer than `need` equal keys at lower indices, or (RANGES)
// inside a forced index range.  A warp takes a tile, lane l ends up with word l of its bits.

// From the bits of the keys beyond the window and the candidates: these set their bits one by one where they are listed, and by words where
// the tile is read again (its 32 keys of a word would take turns at it: 25.6 M equal scores, half of them wanted: 235 us a selection, and 191).
// words: the warp's own [2][32].
__device__ __forceinline__ uint32_t tile_bits(const float *score, size_t P, const SelectWork &w, size_t tile, uint32_t eq_before, uint32_t *words) {
    const uint32_t base = w.state->base, keys = 1u << (20 + w.state->shift), place = w.state->place, need = w.state->need,
                   found = w.tile_found[tile], lane = threadIdx.x & 31u;
    const uint32_t *cand = w.cand + tile * TILE_CANDIDATES + lane;
    const uint32_t c0 = *cand;
    uint32_t bits = tile * MASK_BLOCK + lane * 32u < P ? w.bits[tile * (MASK_BLOCK / 32) + lane] : 0u, equal = 0;
    if (found <= TILE_CANDIDATES) {
        words[lane] = bits;
        words[32 + lane] = 0;
        __syncwarp();
        for_listed(cand, c0, found, [&](bool in, uint32_t c) {
            const uint32_t at = c >> 10;
            if (in && at >= place) atomicOr(words + (at == place ? 32 : 0) + (c >> 5 & 31u), 1u << (c & 31u));
        });
        __syncwarp();
        bits = words[lane];
        equal = words[32 + lane];
    } else {
        for_tile(score, P, tile * MASK_BLOCK, [&](uint32_t w0, const uint32_t (&key)[LOADS], uint32_t left) {
#pragma unroll
            for (int j = 0; j < LOADS; j++) {
                const uint32_t at = window_place(key[j], base);
                const bool in = j * 32u + lane < left && at < keys;
                const uint32_t gt = __ballot_sync(0xffffffffu, in && at > place), eq = __ballot_sync(0xffffffffu, in && at == place);
                if (lane == w0 + j) {
                    bits |= gt;
                    equal = eq;
                }
            }
        });
    }
    if (__any_sync(0xffffffffu, equal != 0)) {
        // the first `need` of all equal keys
        uint32_t before = __popc(equal);
        const uint32_t mine = before;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const uint32_t o = __shfl_up_sync(0xffffffffu, before, d);
            if (lane >= (uint32_t)d) before += o;
        }
        before += eq_before - mine;
        const uint32_t room = need > before ? need - before : 0u;
        for (uint32_t over = mine > room ? mine - room : 0u; over; over--) equal &= ~(0x80000000u >> __clz((int)equal));
        bits |= equal;
    }
    return bits;
}
template <bool RANGES>
__global__ void __launch_bounds__(256)
mask_mark_kernel(const float *score, size_t P, SelectWork w, const uint64_t *ranges, uint32_t nranges,
                 uint32_t *wpre, uint32_t *idx, uint32_t room, uint32_t *tile_sel) {
    __shared__ uint32_t words[8][64];
    if (w.total[1]) return;
    const uint32_t need = w.state->need;
    const uint32_t lane = threadIdx.x & 31u;
    const size_t tile = (size_t)blockIdx.x * 8u + (threadIdx.x >> 5), first = tile * MASK_BLOCK;
    if (first >= P) return;
    const uint64_t run = w.runs[tile / w.run];
    const uint32_t eq_before = w.tile_cand[tile] + (uint32_t)(run >> 32);
    uint32_t bits = tile_bits(score, P, w, tile, eq_before, words[threadIdx.x >> 5]);
    const size_t word = first + lane * 32u;
    if (RANGES) {
        for (uint32_t r = 0; r < nranges; r++) {
            // the part of the range in this word
            const uint64_t lo = ranges[2 * r] > word ? ranges[2 * r] : word, end = word + 32u, hi = ranges[2 * r + 1] < end ? ranges[2 * r + 1] : end;
            if (lo < hi) bits |= (uint32_t)(((1ull << (hi - lo)) - 1ull) << (lo - word));
        }
    }
    if (word < P) w.bits[word >> 5] = bits;
    // positions: what is selected before the tile (the keys above tau and the first `need` of the equal ones), and in the lanes below
    uint32_t at = __popc(bits);
    const uint32_t mine = at;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const uint32_t o = __shfl_up_sync(0xffffffffu, at, d);
        if (lane >= (uint32_t)d) at += o;
    }
    if (RANGES) {
        if (lane == 31) tile_sel[tile] = at;
        return;
    }
    at += w.tile_above[tile] + (uint32_t)run + (eq_before < need ? eq_before : need) - mine;
    if (word < P) wpre[word >> 5] = at;
    // few bits: every lane its own word's; many: all lanes a word's, which are neighbours in the list
    if (__reduce_max_sync(0xffffffffu, mine) <= 12) {
        while (bits) {
            if (at < room) idx[at] = (uint32_t)word + (uint32_t)(__ffs((int)bits) - 1);
            at++;
            bits &= bits - 1u;
        }
    } else {
        const uint32_t below = (1u << lane) - 1u;
#pragma unroll 8
        for (uint32_t l = 0; l < 32; l++) {
            const uint32_t who = __shfl_sync(0xffffffffu, bits, l), to = __shfl_sync(0xffffffffu, at, l) + __popc(who & below);
            if ((who >> lane & 1u) && to < room) idx[to] = (uint32_t)first + l * 32u + lane;
        }
    }
}

cudaError_t launch_mask_mark(const float *score, size_t P, const SelectWork &w, const uint64_t *ranges, uint32_t nranges,
                             uint32_t *wpre, uint32_t *idx, size_t room, uint32_t *tile_sel, cudaStream_t s) {
    const unsigned grid = blocks_for(P, 8 * MASK_BLOCK);
    if (nranges) mask_mark_kernel<true><<<grid, 256, 0, s>>>(score, P, w, ranges, nranges, wpre, idx, (uint32_t)room, tile_sel);
    else mask_mark_kernel<false><<<grid, 256, 0, s>>>(score, P, w, ranges, nranges, wpre, idx, (uint32_t)room, tile_sel);
    return FEDHE_LAUNCHED();
}

// With forced ranges: per-word prefix counts and the ascending index list; a thread takes one word
// of the bit mask (32 parameters), a block the MASK_BLOCK / 32 words of one
// counted block
__global__ void __launch_bounds__(MASK_BLOCK / 32)
mask_write_kernel(size_t P, const uint32_t *bits, const uint32_t *blk_sel_prefix, uint32_t *wpre,
                  uint32_t *idx) {
    __shared__ uint32_t warp_sums[33];
    const size_t word = (size_t)blockIdx.x * (MASK_BLOCK / 32) + threadIdx.x, nwords = (P + 31) >> 5;
    uint32_t w = word < nwords ? bits[word] : 0u;
    uint32_t tot;
    uint32_t before = blk_sel_prefix[blockIdx.x] + block_exclusive_scan((uint32_t)__popc(w), warp_sums, tot);
    if (word < nwords) wpre[word] = before;
    const uint32_t base = (uint32_t)(word << 5);
    while (w) {
        idx[before++] = base + (uint32_t)(__ffs((int)w) - 1);
        w &= w - 1u;
    }
}

cudaError_t launch_mask_write(size_t P, const uint32_t *bits, const uint32_t *blk_sel_prefix,
                              uint32_t *wpre, uint32_t *idx, cudaStream_t s) {
    mask_write_kernel<<<blocks_for(P, MASK_BLOCK), MASK_BLOCK / 32, 0, s>>>(P, bits, blk_sel_prefix, wpre, idx);
    return FEDHE_LAUNCHED();
}

// ===========================================================================
// packing and merging
// ===========================================================================
//
// These are single passes over the update, bound by HBM.  With a mask, a warp
// takes PACK_WORDS consecutive words of the bit mask at a time and lane l the
// parameter of bit l of each: loads and stores of a warp instruction are then
// consecutive addresses (the compacted outputs as well, because the lanes'
// positions are consecutive among the selected / unselected bits of the word),
// and all of a thread's loads are issued before the first store.  Without a
// mask the steps are copies with 16-byte accesses where the pointers allow.

constexpr int PACK_WORDS = 8;       // mask words (256 parameters) per warp
constexpr int COPY_VECS = 4;        // 16-byte vectors per thread of the copies

// masked parameters go to their slot, the others to the compacted remainder.  Bound by HBM now; by its instructions
// while every lane loaded every word and prefix count and had a store for either destination (110 M parameters, 10 %
// masked: 229 us, and 153 us with one load of both and one store, 5.9 TB/s).
__global__ void __launch_bounds__(256)
pack_masked_kernel(const uint32_t *bits, const uint32_t *wpre, const float *x, size_t P, float *sel, float *rest) {
    const uint32_t lane = threadIdx.x & 31u;
    const size_t warp = ((size_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const size_t word0 = warp * PACK_WORDS, nwords = (P + 31) >> 5;
    if (word0 >= nwords) return;
    float v[PACK_WORDS];
#pragma unroll
    for (int j = 0; j < PACK_WORDS; j++) {
        const size_t i = ((word0 + j) << 5) + lane;
        v[j] = i < P ? __ldg(x + i) : 0.0f;
    }
    // the words in lanes 0 .. 7, the counts before them in lanes 8 .. 15
    static_assert(2 * PACK_WORDS <= 32, "a lane for every word and count");
    uint32_t mine = 0;
    if (lane < 2 * PACK_WORDS && word0 + lane % PACK_WORDS < nwords) mine = __ldg((lane < PACK_WORDS ? bits : wpre) + word0 + lane % PACK_WORDS);
#pragma unroll
    for (int j = 0; j < PACK_WORDS; j++) {
        const uint32_t w = __shfl_sync(0xffffffffu, mine, j), pre = __shfl_sync(0xffffffffu, mine, PACK_WORDS + j);
        const size_t i = ((word0 + j) << 5) + lane, before = (size_t)pre + __popc(w & ((1u << lane) - 1u));
        float *dst = (w >> lane) & 1u ? sel + before : rest + (i - before);
        if (i < P) *dst = v[j];
    }
}

// dst[i] = src[i] for i < count, dst[i] = 0 for count <= i < padded (T may be float or double)
template <class T, class V>
__global__ void __launch_bounds__(256)
copy_pad_kernel(const T *src, size_t count, size_t padded, T *dst, bool vec) {
    constexpr size_t per = sizeof(V) / sizeof(T);
    const size_t base = (size_t)blockIdx.x * blockDim.x * COPY_VECS * per;
    if (vec && base + (size_t)blockDim.x * COPY_VECS * per <= count) {
        V t[COPY_VECS];
#pragma unroll
        for (int j = 0; j < COPY_VECS; j++)
            t[j] = __ldg(reinterpret_cast<const V *>(src + base) + j * blockDim.x + threadIdx.x);
#pragma unroll
        for (int j = 0; j < COPY_VECS; j++)
            reinterpret_cast<V *>(dst + base)[j * blockDim.x + threadIdx.x] = t[j];
        return;
    }
    // ragged end of the input, unaligned pointers, and the zero padding
    for (size_t i = base + threadIdx.x; i < base + (size_t)blockDim.x * COPY_VECS * per && i < padded; i += blockDim.x)
        dst[i] = i < count ? src[i] : (T)0;
}

template <class T, class V>
static cudaError_t launch_copy_pad(const T *src, size_t count, size_t padded, T *dst, cudaStream_t s) {
    if (padded == 0) return cudaSuccess;
    const bool vec = ((reinterpret_cast<uintptr_t>(src) | reinterpret_cast<uintptr_t>(dst)) & (sizeof(V) - 1)) == 0;
    const size_t per_block = 256 * COPY_VECS * (sizeof(V) / sizeof(T));
    copy_pad_kernel<T, V><<<blocks_for(padded, (unsigned)per_block), 256, 0, s>>>(src, count, padded, dst, vec);
    return FEDHE_LAUNCHED();
}

__global__ void __launch_bounds__(256) zero_tail_kernel(float *dst, size_t count) {
    const size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < count) dst[i] = 0.0f;
}

cudaError_t launch_pack_range(const he_mask *mask, const float *x, size_t first, size_t count, float *sel, float *rest,
                              cudaStream_t s) {
    if (count == 0) return cudaSuccess;
    const size_t warps = (((count + 31) >> 5) + PACK_WORDS - 1) / PACK_WORDS;
    // positions among the unselected count from the whole mask's start
    pack_masked_kernel<<<blocks_for(warps * 32, 256), 256, 0, s>>>(mask->bits + (first >> 5), mask->wpre + (first >> 5), x, count,
                                                                   sel, rest ? rest + first : nullptr);
    return FEDHE_LAUNCHED();
}

cudaError_t launch_zero(float *dst, size_t count, cudaStream_t s) {
    if (count == 0) return cudaSuccess;
    zero_tail_kernel<<<blocks_for(count, 256), 256, 0, s>>>(dst, count);
    return FEDHE_LAUNCHED();
}

cudaError_t launch_pack(const he_mask *mask, const float *x, size_t P, size_t k, size_t padded,
                        float *sel, float *rest, cudaStream_t s) {
    if (!mask) return launch_copy_pad<float, float4>(x, P, padded, sel, s);     // k = P: a copy and the zero tail
    const cudaError_t e = launch_pack_range(mask, x, 0, P, sel, rest, s);
    if (e) return e;
    return launch_zero(sel + k, padded - k, s);                                  // tail of the last ciphertext
}

// the reverse with a mask: w_glob[i] = z[r] for the r-th masked parameter, the remainder's
// average in order elsewhere
__global__ void __launch_bounds__(256)
unpack_masked_kernel(const uint32_t *bits, const uint32_t *wpre, const double *z, const double *rest_avg, size_t P,
                     double *w_glob) {
    const uint32_t lane = threadIdx.x & 31u;
    const size_t warp = ((size_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const size_t word0 = warp * PACK_WORDS, nwords = (P + 31) >> 5;
    if (word0 >= nwords) return;
    double v[PACK_WORDS];
#pragma unroll
    for (int j = 0; j < PACK_WORDS; j++) {
        const size_t word = word0 + j, i = (word << 5) + lane;
        v[j] = 0.0;
        if (i < P) {
            const uint32_t w = __ldg(bits + word);
            const size_t before = (size_t)__ldg(wpre + word) + __popc(w & ((1u << lane) - 1u));
            v[j] = ((w >> lane) & 1u) ? __ldg(z + before) : __ldg(rest_avg + (i - before));
        }
    }
#pragma unroll
    for (int j = 0; j < PACK_WORDS; j++) {
        const size_t i = ((word0 + j) << 5) + lane;
        if (i < P) w_glob[i] = v[j];
    }
}

cudaError_t launch_unpack_range(const he_mask *mask, const double *z, const double *rest_avg, size_t first, size_t count,
                                double *w_glob, cudaStream_t s) {
    if (count == 0) return cudaSuccess;
    const size_t warps = (((count + 31) >> 5) + PACK_WORDS - 1) / PACK_WORDS;
    unpack_masked_kernel<<<blocks_for(warps * 32, 256), 256, 0, s>>>(mask->bits + (first >> 5), mask->wpre + (first >> 5), z,
                                                                     rest_avg ? rest_avg + first : nullptr, count, w_glob);
    return FEDHE_LAUNCHED();
}

cudaError_t launch_unpack(const he_mask *mask, const double *z, const double *rest_avg, size_t P,
                          double *w_glob, cudaStream_t s) {
    if (P == 0) return cudaSuccess;
    if (!mask) return launch_copy_pad<double, double2>(z, P, P, w_glob, s);
    return launch_unpack_range(mask, z, rest_avg, 0, P, w_glob, s);
}

}  // namespace fedhe

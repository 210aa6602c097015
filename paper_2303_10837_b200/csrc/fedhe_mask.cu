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

// ---- radix selection of the k-th largest key: digits of 11, 10 and 10 bits (a key has 31) ----
//
// Three passes over the scores: the histogram of the first digit; the histogram of the second among the
// keys that have the first (the candidates, a few per cent of real scores), which are also gathered by tiles;
// and, when the threshold tau is known, the marking.  What lies between works on the candidates.  The
// last thread block of a pass to finish does the one-block step that follows it: picking the digit, or
// the scan over the tiles.  (With three histogram passes, a counting pass and one-block kernels between them
// the selection of 2.56 M out of 25.6 M took 341 us; the first pass was bound by conflicts of its shared-memory
// atomics, because neighbouring scores share an exponent.)

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

// Walks the digits of a histogram from the largest down until `need` keys are covered, appends the
// digit found to the prefix and takes the keys above it off `need`.  By a block of 1024 threads.
template <int BITS>
__device__ __forceinline__ void radix_pick(const uint32_t *hist, uint32_t prefix, uint32_t need, SelectState *state) {
    __shared__ uint32_t warp_sums[33];
    constexpr uint32_t bins = 1u << BITS, per = bins / 1024u;        // thread t: digits from bins - 1 - per t down
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
        // the digit where the running count first reaches `need`
        if (above < need && above + h[j] >= need) {
            state->prefix = (prefix << BITS) | (bins - 1u - pos);
            state->need = need - above;
        }
        above += h[j];
    }
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
            if (threadIdx.x == 0) *w.state = SelectState{0xffffffffu, 0u};       // no key reaches the threshold
        } else {
            radix_pick<11>(w.hist, 0u, k, w.state);
        }
    }
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

// Second digit.  A warp takes a tile of MASK_BLOCK scores, counts the keys above the first digit and
// gathers the lower 20 bits of those that have it; a tile with more than TILE_CANDIDATES of them is read again instead.
__global__ void __launch_bounds__(1024, 2)
key_candidates_kernel(const float *score, size_t P, SelectWork w) {
    __shared__ uint32_t sh[1024];
    sh[threadIdx.x] = 0;
    __syncthreads();
    const uint32_t prefix = w.state->prefix, need = w.state->need;
    const uint32_t lane = threadIdx.x & 31u;
    const size_t tiles = (P + MASK_BLOCK - 1) / MASK_BLOCK;
    for (size_t tile = (size_t)blockIdx.x * 32u + (threadIdx.x >> 5); tile < tiles; tile += (size_t)gridDim.x * 32u) {
        const size_t first = tile * MASK_BLOCK;
        uint32_t above = 0, found = 0;
        uint32_t *cand = w.cand + tile * TILE_CANDIDATES;
        for_tile(score, P, first, [&](uint32_t w0, const uint32_t (&key)[LOADS], uint32_t left) {
            // a bit for every candidate among the lane's keys; the few there are get their places together
            uint32_t mine = 0;
#pragma unroll
            for (int j = 0; j < LOADS; j++) {
                const uint32_t top = key[j] >> 20;
                if (top > prefix) above++;
                if (top == prefix) mine |= 1u << j;
            }
            if (left < LOADS * 32u) {                              // keys beyond the end are 0 and not above any digit
                const uint32_t words = left > lane ? (left - lane + 31u) / 32u : 0u;
                mine &= (1u << words) - 1u;
            }
            const uint32_t n = __popc(mine);
            uint32_t at = n;
#pragma unroll
            for (int d = 1; d < 32; d <<= 1) {
                const uint32_t o = __shfl_up_sync(0xffffffffu, at, d);
                if (lane >= (uint32_t)d) at += o;
            }
            const uint32_t all = __shfl_sync(0xffffffffu, at, 31);
            at += found - n;
            found += all;
            while (mine) {
                const uint32_t j = __ffs((int)mine) - 1;
                mine &= mine - 1u;
                const uint32_t low = score_key(__ldg(score + first + (w0 + j) * 32u + lane)) & 0xfffffu;
                if (at < TILE_CANDIDATES) cand[at] = low;
                at++;
                atomicAdd(sh + (low >> 10), 1u);
            }
        });
        above = __reduce_add_sync(0xffffffffu, above);
        if (lane == 0) {
            w.tile_above[tile] = above;
            w.tile_cand[tile] = found;
        }
    }
    __syncthreads();
    if (sh[threadIdx.x]) atomicAdd(w.hist + 2048 + threadIdx.x, sh[threadIdx.x]);
    if (last_block(w.done + 1)) radix_pick<10>(w.hist + 2048, prefix, need, w.state);
}

// f(in, lower 20 bits) for the candidates of a tile, by a whole warp: f may use warp operations
template <class F>
__device__ __forceinline__ void for_candidates(const float *score, size_t P, const SelectWork &w, size_t tile, uint32_t first_digit, F f) {
    const uint32_t lane = threadIdx.x & 31u, found = w.tile_cand[tile];
    if (found <= TILE_CANDIDATES) {
        for (uint32_t i = 0; i < found; i += 32) {
            const bool in = i + lane < found;
            f(in, in ? w.cand[tile * TILE_CANDIDATES + i + lane] : 0u);
        }
    } else {
        for_tile(score, P, tile * MASK_BLOCK, [&](uint32_t, const uint32_t (&key)[LOADS], uint32_t left) {
#pragma unroll
            for (int j = 0; j < LOADS; j++) f(j * 32u + lane < left && (key[j] >> 20) == first_digit, key[j] & 0xfffffu);
        });
    }
}

// third digit, over the candidates
__global__ void __launch_bounds__(1024, 2) key_last_digit_kernel(const float *score, size_t P, SelectWork w) {
    __shared__ uint32_t sh[1024];
    sh[threadIdx.x] = 0;
    __syncthreads();
    const uint32_t prefix = w.state->prefix, need = w.state->need;
    const size_t tiles = (P + MASK_BLOCK - 1) / MASK_BLOCK;
    for (size_t tile = (size_t)blockIdx.x * 32u + (threadIdx.x >> 5); tile < tiles; tile += (size_t)gridDim.x * 32u)
        for_candidates(score, P, w, tile, prefix >> 10, [&](bool in, uint32_t low) {
            if (in && (low >> 10) == (prefix & 1023u)) atomicAdd(sh + (low & 1023u), 1u);
        });
    __syncthreads();
    if (sh[threadIdx.x]) atomicAdd(w.hist + 3072 + threadIdx.x, sh[threadIdx.x]);
    if (last_block(w.done + 2)) radix_pick<10>(w.hist + 3072, prefix, need, w.state);
}

// Keys above and equal to tau: a block takes a run of tiles, and leaves for each the counts before it within the run
// (equal keys in the upper half); the last block does the same for the runs.
__global__ void __launch_bounds__(1024, 2) tile_counts_kernel(const float *score, size_t P, SelectWork w) {
    __shared__ uint64_t warp_sums[33];
    const uint32_t tau = w.state->prefix, need = w.state->need, lane = threadIdx.x & 31u;
    const size_t tiles = (P + MASK_BLOCK - 1) / MASK_BLOCK;
    const size_t begin = (size_t)blockIdx.x * w.run, end = begin + w.run < tiles ? begin + w.run : tiles;
    for (size_t tile = begin + (threadIdx.x >> 5); tile < end; tile += 32u) {
        uint32_t gt = 0, eq = 0;
        for_candidates(score, P, w, tile, tau >> 20, [&](bool in, uint32_t low) {
            gt += in && low > (tau & 0xfffffu) ? 1u : 0u;
            eq += in && low == (tau & 0xfffffu) ? 1u : 0u;
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

cudaError_t launch_select(const float *score, size_t P, size_t k, SelectWork &w, int n_sm, cudaStream_t s) {
    cudaError_t e;
    if ((e = cudaMemsetAsync(w.hist, 0, SELECT_ZEROED * sizeof(uint32_t), s))) return e;
    if ((e = cudaFuncSetAttribute(key_histogram_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)HIST_SMEM))) return e;
    // One thread block of the first pass to an SM, unless its counters could overflow; two keys to a thread are enough (with
    // sixteen, 100 k scores left a thread fourteen loads one after the other: 10 us more).
    const unsigned want = blocks_for(P, 1024 * 2), least = blocks_for(P, (unsigned)HIST_KEYS);
    unsigned g1 = want < (unsigned)n_sm ? want : (unsigned)n_sm;
    if (g1 < least) g1 = least;
    key_histogram_kernel<<<g1, 1024, HIST_SMEM, s>>>(score, P, w, (uint32_t)k);
    if ((e = FEDHE_LAUNCHED())) return e;
    auto grid = [&](unsigned per_block) {
        const unsigned blocks = blocks_for(P, per_block), resident = n_sm < 1024 ? 2u * (unsigned)n_sm : (unsigned)SELECT_RUNS;
        return blocks < resident ? blocks : resident;
    };
    key_candidates_kernel<<<grid(32 * MASK_BLOCK), 1024, 0, s>>>(score, P, w);
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
// inside a forced index range.  A warp takes a tile, a lane the parameter of its number in every word of
// the bit mask.  Without ranges the positions are known, and the prefix counts and the index list are written too.
template <bool RANGES>
__global__ void __launch_bounds__(256)
mask_mark_kernel(const float *score, size_t P, SelectWork w, const uint64_t *ranges, uint32_t nranges, uint32_t *bits,
                 uint32_t *wpre, uint32_t *idx, uint32_t *tile_sel) {
    const uint32_t tau = w.state->prefix, need = w.state->need;
    const uint32_t lane = threadIdx.x & 31u, below = (1u << lane) - 1u;
    const size_t tile = (size_t)blockIdx.x * 8u + (threadIdx.x >> 5), first = tile * MASK_BLOCK;
    if (first >= P) return;
    const uint64_t run = w.runs[tile / w.run];
    uint32_t eq_before = w.tile_cand[tile] + (uint32_t)(run >> 32);
    // selected before the tile: the keys above tau and the first `need` of the equal ones
    uint32_t at = RANGES ? 0u : w.tile_above[tile] + (uint32_t)run + (eq_before < need ? eq_before : need);
    // lane l keeps the bits and the prefix count of word l of the tile, which are stored together
    uint32_t my_bits = 0, my_pre = 0;
    static_assert(MASK_BLOCK == 1024, "a word of the tile for every lane");
    for_tile(score, P, first, [&](uint32_t w0, const uint32_t (&key)[LOADS], uint32_t left) {
        bool equal = false;
#pragma unroll
        for (int j = 0; j < LOADS; j++) equal = equal || key[j] == tau;
        // keys equal to tau are rare (among real scores), and keys beyond the end are 0
        const bool some = __any_sync(0xffffffffu, equal);
#pragma unroll
        for (int j = 0; j < LOADS; j++) {
            const uint32_t i = (uint32_t)first + (w0 + j) * 32u + lane;        // parameters are fewer than 2^32
            bool sel = key[j] > tau;
            if (some || RANGES) {
                const bool in = j * 32u + lane < left, eq = in && key[j] == tau;
                const uint32_t eqs = __ballot_sync(0xffffffffu, eq);
                sel = sel || (eq && eq_before + __popc(eqs & below) < need);
                eq_before += __popc(eqs);
                if (RANGES && in && !sel)
                    for (uint32_t r = 0; r < nranges; r++)
                        if (i >= ranges[2 * r] && i < ranges[2 * r + 1]) sel = true;
            }
            const uint32_t who = __ballot_sync(0xffffffffu, sel);
            if (lane == w0 + j) {
                my_bits = who;
                my_pre = at;
            }
            if (!RANGES && sel) idx[at + __popc(who & below)] = i;
            at += __popc(who);
        }
    });
    if (first + lane * 32u < P) {
        bits[(first >> 5) + lane] = my_bits;
        if (!RANGES) wpre[(first >> 5) + lane] = my_pre;
    }
    if (RANGES && lane == 0) tile_sel[tile] = at;
}

cudaError_t launch_mask_mark(const float *score, size_t P, const SelectWork &w, const uint64_t *ranges, uint32_t nranges,
                             uint32_t *bits, uint32_t *wpre, uint32_t *idx, uint32_t *tile_sel, cudaStream_t s) {
    const unsigned grid = blocks_for(P, 8 * MASK_BLOCK);
    if (nranges) mask_mark_kernel<true><<<grid, 256, 0, s>>>(score, P, w, ranges, nranges, bits, wpre, idx, tile_sel);
    else mask_mark_kernel<false><<<grid, 256, 0, s>>>(score, P, w, ranges, nranges, bits, wpre, idx, tile_sel);
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

// masked parameters go to their slot, the others to the compacted remainder
__global__ void __launch_bounds__(256)
pack_masked_kernel(const uint32_t *bits, const uint32_t *wpre, const float *x, size_t P, float *sel, float *rest) {
    const uint32_t lane = threadIdx.x & 31u;
    const size_t warp = ((size_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const size_t word0 = warp * PACK_WORDS, nwords = (P + 31) >> 5;
    if (word0 >= nwords) return;
    float v[PACK_WORDS];
    uint32_t w[PACK_WORDS], pre[PACK_WORDS];
#pragma unroll
    for (int j = 0; j < PACK_WORDS; j++) {
        const size_t word = word0 + j, i = (word << 5) + lane;
        v[j] = i < P ? __ldg(x + i) : 0.0f;
        w[j] = word < nwords ? __ldg(bits + word) : 0u;
        pre[j] = word < nwords ? __ldg(wpre + word) : 0u;
    }
#pragma unroll
    for (int j = 0; j < PACK_WORDS; j++) {
        const size_t i = ((word0 + j) << 5) + lane;
        if (i >= P) continue;
        const size_t before = (size_t)pre[j] + __popc(w[j] & ((1u << lane) - 1u));
        if ((w[j] >> lane) & 1u) sel[before] = v[j];
        else rest[i - before] = v[j];
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

// Internal types shared by the kernels and the C ABI of the CUDA library.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <vector>

#include "../../include/fedhe.h"
#include "fedhe_fft.cuh"
#include "fedhe_host.h"
#include "fedhe_ntt.cuh"

namespace fedhe {

// How a centred residue is cut: v = sum_p piece_p 2^shift_p, p < pieces.
struct FftSplit {
    uint32_t pieces, shift[FFT_MAX_PIECES];
    uint32_t narrow;     // two pieces, and the rounded product of the lower one fits 32 bits
    double top_scale;    // 2^(shift of the top piece) / q
};

// Cuts a centred residue (|v| < q/2) into its pieces, lowest first; each but the top one lies in
// [-2^(w-1), 2^(w-1)) for its width w.
HD int64_t fft_piece(const FftSplit &f, int64_t v, uint32_t p) {
    for (uint32_t i = 0; i + 1 < f.pieces; i++) {
        const uint32_t w = f.shift[i + 1] - f.shift[i];
        const int64_t up = (v + ((int64_t)1 << (w - 1))) >> w;
        if (i == p) return v - (int64_t)((uint64_t)up << w);
        v = up;
    }
    return v;
}

// What an encryption computes together: a limb, by the products of its pieces from the lowest to the top one, or
// two limbs whose low pieces are a few bits wide, by one product of both of them, the first's plus 2^16 times
// the second's, and their top ones.
constexpr uint32_t NO_LIMB = 0xffffffffu;
struct EncUnit {
    uint32_t limb, limb2;        // limb2 = NO_LIMB: a single one
    uint32_t products;
    size_t fft_key;              // first word of its key tables: [2 components][products][n]
};
// The units of a public-key half.
struct EncWay {
    uint32_t units, products;    // of all units
    EncUnit unit[HE_MAX_LIMBS];
};
// Its products, in the order in which a thread block works them off: a low piece's is parked, a top one's ends its limb.
struct alignas(16) EncJob {
    uint64_t q;
    double scale;                // of the limb's quotients
    uint32_t key[2];             // blocks of 2^12 words before the key tables, for either component
    uint32_t shift;              // the top piece's
    uint32_t what;               // limb (of the low product of a pair: of the first of them), flags, and above them what is parked for
                                 // a top piece: 0 nothing, 1 its low piece's product, 2, 3 that of a pair, lower or upper limb
    static constexpr uint32_t PARKS = 1u << 8, NARROW = 1u << 9, JOINS = 10;
};
struct alignas(16) EncJobs {
    EncJob job[2 * HE_MAX_LIMBS];
    uint8_t start[4 * HE_MAX_LIMBS + 1];       // of the products of both components: the first at or after a number that begins a unit
};
// Limbs in pairs where that is possible, and, if any are, every limb by itself too: fewer products, or more units to share out.
constexpr uint32_t ENC_MOST = 8;       // thread blocks of a cluster that encrypts, at most
constexpr uint32_t ENC_SHARES = 2 * HE_MAX_LIMBS + ENC_MOST;
struct EncWays {
    uint32_t count;
    EncWay way[2];
    EncJobs jobs[2];
    uint16_t most[2][ENC_SHARES];      // of the products of a ciphertext shared out to so many blocks, the most that one has
};

// Per-prime constants and table pointers, passed to kernels by value.
struct LimbDev {
    uint64_t q;          // the prime
    uint64_t mu;         // floor(2^64 / q), Barrett
    tw_t ninv;           // 1/N
    tw_t wn;             // (inverse twiddle of stage 0) / N
    tw_t r64;            // 2^64 mod q
    tw_t qlinv;          // 1 / q_{L-1} mod q (unused for the last prime)
    const tw_t *fwd;     // psi^brev(i)
    const tw_t *inv;     // psi^-brev(i)
    // primes below F64_PRIME_LIMIT also carry what the double-precision
    // transforms need (fwd_d is null for the others)
    const double *fwd_d; // the same twiddles as doubles
    const double *inv_d;
    double qd, qi;       // q and 1/q rounded
    double ninv_d, wn_d; // 1/N and (inverse twiddle of stage 0)/N
    FftSplit split[2];   // of the public key's residues: for a limb by itself, and where limbs go in pairs
};

// the pieces of a limb that a transform in arithmetic M needs
template <class M>
struct LimbOf;
template <bool SEL>
struct LimbOf<ModIntT<SEL>> {
    static HD NttArgsT<ModIntT<SEL>> args(const LimbDev &lb, bool fwd, uint32_t A, uint32_t blk) {
        return NttArgsT<ModIntT<SEL>>{fwd ? lb.fwd : lb.inv, ModIntT<SEL>{lb.q, 2 * lb.q}, A, blk};
    }
    static HD tw_t ninv(const LimbDev &lb) { return lb.ninv; }
    static HD tw_t wn(const LimbDev &lb) { return lb.wn; }
};
template <>
struct LimbOf<ModF64> {
    static HD NttArgsF args(const LimbDev &lb, bool fwd, uint32_t A, uint32_t blk) {
        return NttArgsF{fwd ? lb.fwd_d : lb.inv_d, ModF64{lb.qd, lb.qi}, A, blk};
    }
    static HD double ninv(const LimbDev &lb) { return lb.ninv_d; }
    static HD double wn(const LimbDev &lb) { return lb.wn_d; }
};

struct CtxDev {
    uint32_t N, logN, L;
    uint32_t LOGB, A;    // a length-N transform = 2^A blocks of 2^LOGB
    int32_t log2_delta;
    LimbDev limb[HE_MAX_LIMBS];
    const LimbDev *limb_dev;   // the same table in device memory, for kernels that loop over limbs
    const double2 *ftw;  // slot-transform twiddles, entry [len/2 + j]
    const root_t *fft_fwd, *fft_inv;   // complex transforms of the exact products (fedhe_fft.cuh)
    const uint32_t *slot_of;           // slot of every value that the forward transform leaves
    FftSplit dec_split;                // of c1 on limb 0, for any c1
    const EncWays *enc;                // host memory (the context's): kernels get the way they take by value
    const EncJobs *enc_jobs;           // of either way, in device memory
    int64_t term_limit;                // a quarter of the smallest prime
    uint16_t enc_fit[2][ENC_MOST + 1]; // clusters of a size that the device holds: two blocks to an SM, one
    uint32_t passes_most;              // encryption by passes (N = 2^16): the most ciphertexts that go by them
    const void *gauss;   // GaussTables
    uint32_t sm_count;
    uint32_t *deal;      // encryption hands out ciphertexts here: next one, thread blocks (clusters) that are done; 0 between calls
    int *status;         // sticky anomaly word
};

struct KeysDev {
    const tw_t *pk0_hat; // [L][N] transform-domain public key with Shoup companions
    const tw_t *pk1_hat;
    const tw_t *s_hat;   // [L][N] transform-domain secret key
    const int8_t *s;     // [N]
    const double2 *fft_pk; // transformed pieces of the public key, scaled by 1/n, in the threads' order
    const double2 *fft_s;  // the transformed secret key in the same order and scale
};

}  // namespace fedhe

struct he_ctx {
    uint32_t magic;
    int device;
    fedhe::CtxDev dev;
    fedhe::EncWays enc;
    he_params params;
    std::vector<void *> owned;     // device allocations freed with the context
    // growable work buffers (device)
    void *ws = nullptr;            // encode output / decrypt scratch
    size_t ws_bytes = 0;
    void *tab = nullptr;           // per-call pointer and weight tables
    size_t tab_bytes = 0;
    void *round_buf = nullptr;     // buffers of he_round_host
    size_t round_bytes = 0;
    int sm_count = 0;
    cudaStream_t copy_stream = nullptr;   // uploads of he_round_host, overlapped with compute
    cudaStream_t down_stream = nullptr;   // downloads of he_round_host (PCIe carries both directions at once)
    cudaEvent_t ev_ready[2] = {nullptr, nullptr}, ev_free[2] = {nullptr, nullptr};
    cudaEvent_t ev_chunk = nullptr;       // a chunk's result is ready for download
};

struct he_keys {
    uint32_t magic;
    he_ctx *ctx;
    fedhe::KeysDev dev;
    void *storage;
    bool is_share = false;   // a party's share of the secret (no public key, no small secret)
};

struct he_mask {
    uint32_t magic;
    int device;
    size_t P, k;
    uint32_t *idx;       // [k] ascending
    uint32_t *bits;      // [ceil(P/32)] bit i of word i/32 set if parameter i is encrypted
    uint32_t *wpre;      // [ceil(P/32)] number of encrypted parameters before the word
};

namespace fedhe {
constexpr uint32_t CTX_MAGIC = 0x48454358u, KEYS_MAGIC = 0x48454b59u, MASK_MAGIC = 0x48454d4bu;
}

// Launch wrappers of the CUDA kernels (implemented in fedhe_transform.cu, fedhe_slots.cu, fedhe_encrypt.cu, fedhe_fft.cu, fedhe_server.cu, fedhe_decrypt.cu and fedhe_mask.cu),
// called by the C ABI in fedhe_api.cu.  All of them enqueue work on `s` and
// return the launch status; none synchronises.
#pragma once

#include "fedhe_internal.cuh"

namespace fedhe {

uint64_t launch_count();

// In-place negacyclic transforms of `npoly` polynomials.  Polynomial p, limb
// l (0 <= l < nlimbs, using prime limb0 + l) starts at data + p*poly_stride
// + l*N.  Forward input may lie in [0, 4q), inverse input in [0, 2q);
// outputs are canonical.
cudaError_t launch_ntt(const CtxDev &c, bool forward, uint64_t *data, size_t npoly, size_t poly_stride,
                       uint32_t limb0, uint32_t nlimbs, cudaStream_t s);

// keygen pieces: tmp is uint64 [3][L][N]
cudaError_t launch_keygen_sample(const CtxDev &c, uint64_t seed, int8_t *s8, uint64_t *tmp, cudaStream_t s);
cudaError_t launch_keygen_combine(const CtxDev &c, const uint64_t *tmp, tw_t *pk0_hat, tw_t *pk1_hat,
                                  tw_t *s_hat, cudaStream_t s);
cudaError_t launch_extract_values(const tw_t *src, uint64_t *dst, size_t count, cudaStream_t s);

// slot transform.  cplx: scratch of T*n double2, used only when n > 8192
cudaError_t launch_encode(const CtxDev &c, const float *sel, size_t T, double2 *cplx, int64_t *m,
                          cudaStream_t s);
cudaError_t launch_decode(const CtxDev &c, const int64_t *d, size_t T, double2 *cplx, double *z,
                          cudaStream_t s);

// Encode + encrypt ciphertexts t0 .. t0+T-1 (sel and ct point at the first of
// them).  `work` is scratch of fft_work_bytes() bytes: the random draws (for 256 MiB
// of them at a time) and what the resident thread blocks keep in L2, or, by passes, what those need.
size_t fft_work_bytes(const CtxDev &c, size_t T);
cudaError_t launch_encrypt(const CtxDev &c, const KeysDev &k, const float *sel, void *work, uint32_t t0, size_t T,
                           uint64_t seed, uint32_t client, uint64_t *ct, cudaStream_t s);
// Once per context: how the products cut the residues (from the primes); then, on its device, what the device holds of these kernels (CtxDev::enc_fit).
bool fft_cut(CtxDev &c, EncWays &e);
size_t fft_key_words(const CtxDev &c);
cudaError_t fft_setup(CtxDev &c, int n_sm);
// The same by passes over the ciphertext, on the longest ring, for the numbers of ciphertexts where encrypt_by_passes() says that it
// is faster; scratch of encrypt_passes_work_bytes() for any number up to T (16 N bytes for each that may go by passes).
constexpr uint32_t PASSES_KNOWN = 1024;
bool encrypt_by_passes(const CtxDev &c, size_t T);
uint32_t passes_most(const CtxDev &c);                // sets CtxDev::passes_most
double enc_transforms_us(const CtxDev &c, size_t T);   // estimate of the time by transforms
size_t encrypt_passes_work_bytes(const CtxDev &c, size_t T);
cudaError_t launch_encrypt_passes(const CtxDev &c, const KeysDev &k, const float *sel, void *work, uint32_t t0, size_t T,
                                  uint64_t seed, uint32_t client, uint64_t *ct, cudaStream_t s);
// Decrypt + decode T coefficient-domain ciphertexts; by launch_decrypt() and launch_decode() where decrypt_by_passes() says that
// those are faster.
bool decrypt_by_passes(const CtxDev &c, size_t T);
cudaError_t launch_decrypt_fft(const CtxDev &c, const KeysDev &k, const uint64_t *ct, uint32_t level, size_t T,
                               double *z, cudaStream_t s);
// The table of the discrete Gaussian that encryption reads (CtxDev::gauss).
size_t gauss_table_bytes();
cudaError_t launch_gauss_table(void *table, cudaStream_t s);
// Key tables of both from the public key's coefficients ([2][L][N], canonical) and the secret.
cudaError_t launch_fft_keys(const CtxDev &c, const uint64_t *pk, const int8_t *s8, double2 *fft_pk, double2 *fft_s,
                            cudaStream_t s);

// Encryption with every limb polynomial of the result in the transform domain; `work`: for N <= 2^14
// N words per thread block of the fused kernel (the block's encoded message), for longer rings the
// encoded messages of all T ciphertexts, the encoder's complex buffer and the transform of u.
size_t encrypt_ntt_work_bytes(const CtxDev &c, int n_sm, size_t T);
cudaError_t launch_encrypt_ntt(const CtxDev &c, const KeysDev &k, const float *sel, void *work, int n_sm,
                               uint32_t t0, size_t T, uint64_t seed, uint32_t client, uint64_t *ct,
                               cudaStream_t s);

// What a weighted sum needs to know of C clients: their C pointers, then what they are weighed by ([C][L] tw_t for ciphertexts, [C]
// doubles for the remainder).  A small table goes with the kernel's parameters: a copy to the device from memory that is not pinned
// costs the call 2 us on the host and makes the kernel wait for it (25 ciphertexts of N = 8192, three limbs, copied and not: 3 clients, 21 words,
// 14.5 and 12.4 us; 9, 63 words, 26.8 and 24.8; 18, 126 words, 43.9 and 42.9).  A larger one is copied: threads that read different words of the
// parameters take turns, and what is gained is lost again (32 clients, 224 words, 66.6 and 66.5; 64, 448 words, 120.4 and 121.9).
struct SumTable {
    static constexpr size_t WORDS = 128;
    const uint64_t *far;                  // in device memory; null: here
    uint64_t words[WORDS];
};
// `words` words of the host to device memory, as parameters of kernels that write them
cudaError_t launch_table(const void *host, size_t words, uint64_t *dst, cudaStream_t s);
cudaError_t launch_aggregate(const CtxDev &c, const SumTable &tab, int C,
                             size_t T, uint64_t *out, int n_sm, cudaStream_t s);
// transform-domain ciphertexts in and out; scratch: uint64 [T][2][L][N]
cudaError_t launch_aggregate_ntt(const CtxDev &c, const SumTable &tab, int C,
                                 size_t T, uint64_t *scratch, uint64_t *out, int n_sm, cudaStream_t s);
// aligned16: every client's pointer is 16-byte aligned (the caller knows the host copies)
// the clients' weighted sum on all L limbs without the rescale, and the rescale of a sum of such sums
cudaError_t launch_aggregate_partial(const CtxDev &c, const SumTable &tab, int C,
                                     size_t T, uint64_t *out, int n_sm, cudaStream_t s);
cudaError_t launch_rescale_partial_sum(const CtxDev &c, const uint64_t *const *parts, int P, size_t T,
                                       uint64_t *out, cudaStream_t s);
cudaError_t launch_plain_aggregate(const SumTable &tab, int C, size_t len,
                                   double *out, bool aligned16, cudaStream_t s);

// scratch: uint64 [T][N]; on return it holds the centred integers as int64
cudaError_t launch_decrypt(const CtxDev &c, const KeysDev &k, const uint64_t *ct, uint32_t level,
                           size_t T, uint64_t *scratch, cudaStream_t s);

// the same for a transform-domain ciphertext
cudaError_t launch_decrypt_ntt(const CtxDev &c, const KeysDev &k, const uint64_t *ct, uint32_t level,
                               size_t T, uint64_t *scratch, cudaStream_t s);

// fused decrypt + decode of a transform-domain ciphertext for N <= 2^14 (no scratch): z double [T][n]
cudaError_t launch_decrypt_ntt_fused(const CtxDev &c, const KeysDev &k, const uint64_t *ct, uint32_t level,
                                     size_t T, double *z, cudaStream_t s);

// two-party threshold decryption.  tmp: uint64 [2][L][N] (shares as residues)
cudaError_t launch_threshold_split(const CtxDev &c, const int8_t *s8, uint64_t seed, uint64_t *tmp,
                                   cudaStream_t s);
cudaError_t launch_share_tables(const CtxDev &c, const uint64_t *share_hat, tw_t *s_hat, cudaStream_t s);
// part: uint64 [T][N], work space and result (canonical residues mod q_0)
cudaError_t launch_partial_decrypt(const CtxDev &c, const KeysDev &share, uint32_t party, const uint64_t *ct,
                                   uint32_t level, size_t T, uint64_t seed, uint32_t bits, uint64_t *part,
                                   cudaStream_t s);
struct PartPtrs { const uint64_t *p[8]; };
cudaError_t launch_threshold_combine(const CtxDev &c, const uint64_t *ct, uint32_t level, const PartPtrs &parts,
                                     int nparts, size_t T, int64_t *d, cudaStream_t s);

// context-owned work space for T ciphertexts (2 * T * N words); implemented in fedhe_api.cu
int ctx_workspace(he_ctx *ctx, size_t T, void **out);

// mask construction (tiles of MASK_BLOCK consecutive parameters)
constexpr uint32_t MASK_BLOCK = 1024, TILE_CANDIDATES = 128;
// progress of the selection, in device memory: the window [base, base + 2^(20 + shift)) of keys that the threshold is looked for in, how much
// of its place in there is found (all of it after the last step: tau = base + place), and how many keys are still to be covered
// (after the last step: how many keys equal to tau belong to the mask)
struct SelectState { uint32_t base, shift, place, need, above; };      // above: keys beyond the window
constexpr uint32_t WINDOW_OPEN = 3;               // shift: the sample could not say
// work space of a selection; the words from `hist` to the end of `sampled` are cleared at its start
constexpr size_t SELECT_LAST = 4096, SELECT_HIST = 2048 + 1024 + SELECT_LAST, SELECT_BINS = 1u << 12, SELECT_ZEROED = SELECT_HIST + 8 + 8;
constexpr size_t SELECT_RUNS = 2 * 1024;          // thread blocks that a device holds at once, at most
struct SelectWork {
    uint32_t *hist;              // 2048, 1024, SELECT_LAST
    uint32_t *done;              // [5] thread blocks that finished a pass
    SelectState *state;
    uint32_t *total;             // selected parameters (without forced ranges), then whether the threshold was outside the window
    uint32_t *sampled;           // [SELECT_BINS] keys of the sample by their upper bits
    uint32_t *tile_above, *tile_cand, *tile_found, *cand;     // per tile; [tiles][TILE_CANDIDATES]
    uint64_t *runs;              // [SELECT_RUNS] counts before a run of tiles
    uint32_t run;                // tiles of a run (set by launch_select)
    uint32_t *bits;              // the mask's: the keys beyond the window are marked by the pass that looks for candidates
};
// whether a sample may choose the window (without forced ranges); it can miss, and total[1] is not 0 then
bool select_by_sample(size_t P, size_t k);
cudaError_t launch_select(const float *score, size_t P, size_t k, bool by_sample, SelectWork &w, int n_sm, cudaStream_t s);
// in-place exclusive scan of a[0..count); the grand total goes to *total
cudaError_t launch_scan(uint32_t *a, size_t count, uint32_t *total, cudaStream_t s);
cudaError_t launch_mask_mark(const float *score, size_t P, const SelectWork &w, const uint64_t *ranges, uint32_t nranges,
                             uint32_t *wpre, uint32_t *idx, size_t room, uint32_t *tile_sel, cudaStream_t s);      // idx holds `room`
cudaError_t launch_mask_write(size_t P, const uint32_t *bits, const uint32_t *blk_sel_prefix,
                              uint32_t *wpre, uint32_t *idx, cudaStream_t s);

// the same for the parameters [first, first + count) of a mask, first a multiple of 32: x and w_glob point at the first
// of them, sel, rest, z and rest_avg at the start of the whole arrays
cudaError_t launch_pack_range(const he_mask *mask, const float *x, size_t first, size_t count, float *sel, float *rest,
                              cudaStream_t s);
cudaError_t launch_unpack_range(const he_mask *mask, const double *z, const double *rest_avg, size_t first, size_t count,
                                double *w_glob, cudaStream_t s);
cudaError_t launch_zero(float *dst, size_t count, cudaStream_t s);
cudaError_t launch_pack(const he_mask *mask, const float *x, size_t P, size_t k, size_t padded,
                        float *sel, float *rest, cudaStream_t s);
cudaError_t launch_unpack(const he_mask *mask, const double *z, const double *rest_avg, size_t P,
                          double *w_glob, cudaStream_t s);

}  // namespace fedhe

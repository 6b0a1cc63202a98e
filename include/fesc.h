/*
 * fesc.h -- C ABI of the B200 (sm_100a) RNS-CKKS linear hot path used by FESC's
 * encrypted Mamba-2 inference: negacyclic NTT, ciphertext x plaintext
 * multiply-accumulate, Galois rotation with hybrid (dnum) key switching (plain, hoisted,
 * rotate-and-add), rescale, ciphertext x ciphertext products, the BSGS plaintext-weight
 * projection, the causal depthwise convolution, the real / imaginary split of complex-packed
 * results and the factorized scan-contract.
 *
 * Conventions shared by every call
 *   - All residues are uint64 in [0, q) ("canonical").  Polynomials are stored limb by
 *     limb, N contiguous words per limb.  "EVAL" form is the bit-reversed evaluation
 *     order  EVAL[t] = sum_i COEFF[i] * psi^((2*brev(t)+1)*i) mod q  with psi the smallest
 *     primitive 2N-th root of unity modulo q.
 *   - A ciphertext at level l (l active data limbs) is [2][l][N]: c0 then c1, EVAL form.
 *     A batch is [batch][2][l][N].  Limb i of a ciphertext uses data prime i.
 *   - Pointers named `d_*` or documented "device" are device pointers owned by the
 *     caller; the library never frees or reallocates them.  Arrays of words need the
 *     alignment of a word (8 bytes; 16 are faster), a packed image (below) 16 bytes:
 *     FESC_EINVAL otherwise.  `stream` is a cudaStream_t
 *     passed as void* (NULL = default stream).  Calls enqueue work on `stream` and return
 *     without synchronising, unless stated otherwise.
 *   - Scratch memory belongs to the context.  It grows (cudaFree + cudaMalloc, which
 *     synchronises the device) the first time a call needs more than is reserved; calls
 *     with sizes already seen allocate nothing.  One context must not be used from two
 *     streams at the same time (the scratch is shared).
 *   - Return value: FESC_OK (0) or a negative FESC_E* code; fesc_last_error() gives text.
 *     Asynchronous CUDA errors surface at a later call or at fesc_sync().
 *
 * The paper treats its CKKS backend as a black box (Sec. 8.1 "FHE Settings"); the
 * primitive list is its Table "CKKS primitives" (add, ptmul, ctmul, rot, conj), the
 * projection is App. "Projection Kernel Breakdown", the scan-contract is Sec. 5.4
 * (Eqs. fesc_recurrence / fesc_contract).
 */
#ifndef FESC_H
#define FESC_H

#include <stddef.h>
#include <stdint.h>

#ifdef __cplusplus
extern "C" {
#endif

typedef struct fesc_ctx fesc_ctx;

enum {
    FESC_OK = 0,
    FESC_EINVAL = -1,   /* bad argument (sizes, non-prime or non NTT-friendly modulus, ...) */
    FESC_ENOMEM = -2,   /* host or device allocation failed */
    FESC_ECUDA = -3,    /* a CUDA runtime call failed */
    FESC_ELEVEL = -4,   /* level out of range for the operation (e.g. rescale at level 1) */
    FESC_ENOKEY = -5,   /* no evaluation key registered under the given key id */
    FESC_ETIMEOUT = -6, /* a bounded device-side wait on an asynchronous copy gave up; reported by fesc_sync */
    FESC_EBOUNDS = -7   /* debug build only: a kernel skipped a region outside every known extent; reported by fesc_sync */
};

/* "rotation amount" that selects complex conjugation instead of a slot rotation */
#define FESC_CONJ INT32_MIN
/* key id reserved for the relinearisation key generated by fesc_ctx_create */
#define FESC_RELIN_KEY_ID 0u

/*
 * The CKKS backend below (RNS residues, NTT, hybrid key switching, rescale) is the standard construction the paper
 * assumes in Sec. 2 "Fully Homomorphic Encryption and CKKS" and configures in Sec. 8.1 "FHE Settings".
 *
 * Create a context: ring degree N = 2^log_n (log_n in [4,12] or 16), `n_q` data primes
 * followed by `n_p` special primes in `primes` (HOST array, each prime = 1 mod 2N and
 * < 2^62), key-switch digit count `dnum` (alpha = ceil(n_q/dnum) limbs per digit).
 * Builds the twiddle and basis-conversion tables, the ternary secret key and the
 * relinearisation key, all derived from `seed` with the counter-based generator
 *   word(seed, tag, index) = M(M(seed ^ M(tag)) + index),
 *   M(z): z += 0x9E3779B97F4A7C15; z = (z ^ z>>30) * 0xBF58476D1CE4E5B9;
 *         z = (z ^ z>>27) * 0x94D049BB133111EB; return z ^ z>>31,
 *   tag = domain | key_id<<8 | digit<<40 | limb<<48
 * (secret: domain 1, ternary floor(3*word/2^64)-1; key masks a: domain 2, uniform
 * floor(word*q/2^64), drawn in EVAL form; key errors e: domain 3, centred binomial
 * popcount(word & (2^21-1)) - popcount((word>>21) & (2^21-1))).  This generator is for
 * reproducible benchmarking, not for protecting data.
 * Switching keys follow the hybrid construction: for digit j and every modulus t,
 *   b_j = -a_j s + e_j + [t in digit j] (P mod q_t) s',  stored as [digit][b,a][n_q+n_p][N].
 * Synchronises the device.  Errors: FESC_EINVAL, FESC_ENOMEM, FESC_ECUDA.
 */
int fesc_ctx_create(fesc_ctx** out, uint32_t log_n, const uint64_t* primes, uint32_t n_q,
                    uint32_t n_p, uint32_t dnum, uint64_t seed);
int fesc_ctx_destroy(fesc_ctx* ctx);

/*
 * Derived parameters of a context, or of a parameter set before any context exists (fesc_params_info runs on the
 * host alone and needs no GPU).  Hybrid key switching (Sec. 2 "Fully Homomorphic Encryption and CKKS") adds noise of
 * about Q_j / P times the key error per digit, so a parameter set whose special modulus P is smaller than the largest
 * digit modulus Q_j = product of a digit's primes switches keys with noise above the message scale: such a set is
 * accepted (its residues are still well defined and bit-exact) but flagged with FESC_INFO_KEYSWITCH_NOISE.
 */
typedef struct fesc_info {
    uint32_t log_n, n_q, n_p, dnum;
    uint32_t alpha;        /* limbs per key-switch digit, ceil(n_q / dnum) */
    uint32_t digits;       /* key-switch digits at full level, ceil(n_q / alpha) */
    uint32_t flags;        /* FESC_INFO_* */
    uint32_t reserved;
    double log2_P;         /* log2 of the special modulus */
    double log2_Qmax;      /* log2 of the largest digit modulus */
} fesc_info;
#define FESC_INFO_KEYSWITCH_NOISE 1u   /* P < max_j Q_j: rotations and products decrypt with noise above the scale */
int fesc_params_info(uint32_t log_n, const uint64_t* primes, uint32_t n_q, uint32_t n_p, uint32_t dnum, fesc_info* out);
int fesc_ctx_info(const fesc_ctx* ctx, fesc_info* out);
/* Test hook (no counterpart in the paper): the next `count` scratch-arena allocations of this context report
 * FESC_ENOMEM without calling the driver, so that callers can exercise their handling of allocation failure. */
int fesc_ctx_test_fail_allocs(fesc_ctx* ctx, uint32_t count);
/* Bounds-checking debug build (no counterpart in the paper; a development aid where a memory checker cannot be run).
 * The library built with -DFESC_DEBUG_BOUNDS (libfesc_b200_dbg.so) makes every kernel compare the regions it is about
 * to touch with a table of extents: the library's own allocations plus the caller's buffers registered here.  A
 * region outside every extent is not touched; it is counted and the first one recorded, and the next fesc_sync
 * returns FESC_EBOUNDS with file id, line, address and size in fesc_last_error.  Nothing traps and the context stays
 * usable.  The table is per process (one device), holds the 192 caller buffers registered most recently, and a buffer registered
 * again at the same address takes the new size.  d_ptr: device pointer; bytes: its extent.  _report copies the count
 * of skipped regions and the first record to host words (any may be NULL) and starts a new record.
 * In the release library all three return FESC_EINVAL. */
int fesc_debug_bounds_register(const void* d_ptr, size_t bytes);
int fesc_debug_bounds_clear(void);
int fesc_debug_bounds_report(uint32_t* hits, uint32_t* first_site, uint64_t* first_addr, uint64_t* first_bytes);
/* Give the context's scratch arena back to the device (synchronises the device); the next call that needs scratch
 * reserves it again.  For callers that alternate between workloads with very different scratch needs. */
int fesc_ctx_trim(fesc_ctx* ctx);
/* Text of the last error recorded on this context (never NULL). */
const char* fesc_last_error(const fesc_ctx* ctx);
/* Wait for `stream` and report any pending CUDA error, or FESC_ETIMEOUT if a kernel's bounded wait gave up. */
int fesc_sync(fesc_ctx* ctx, void* stream);

/*
 * Self-test of the library's bounded device-side waits (no counterpart in the paper): launches one warp that waits
 * on a barrier phase nothing completes, with a budget of 4096 polls; the wait runs out, the kernel records it in the
 * context's status word and returns.  The next fesc_sync on the stream returns FESC_ETIMEOUT (and clears the word);
 * the context stays usable.  Nothing faults, traps or hangs.
 */
int fesc_selftest_wait_limit(fesc_ctx* ctx, void* stream);

/*
 * Generate and register the Galois key for the slot rotation rho(v; rot)_j = v_{(j+rot) mod n}
 * (Sec. 5.1; cyclic LEFT shift, g = 5^rot mod 2N) or, with rot == FESC_CONJ, for complex
 * conjugation (g = 2N-1), under `key_id` (1 .. 2^24-1; re-registering an id replaces it).
 * Allocates (n_digits * 2 * (n_q+n_p) * N) words of device memory owned by the context.
 * Synchronises the device.
 */
int fesc_ctx_add_galois_key(fesc_ctx* ctx, int32_t rot, uint32_t key_id);
/* Copy a registered key ([digit][2][n_q+n_p][N] words) or the secret key in EVAL form
 * ([n_q+n_p][N] words) to a DEVICE buffer; for tests of the key generator. */
int fesc_ctx_export_key(fesc_ctx* ctx, uint32_t key_id, uint64_t* d_dst, void* stream);
int fesc_ctx_export_secret(fesc_ctx* ctx, uint64_t* d_dst, void* stream);
/* Number of key-switch digits at full level, ceil(n_q / alpha). */
uint32_t fesc_ctx_num_digits(const fesc_ctx* ctx);
/* Counters since creation: [0] limb transforms, [1] key switches, [2] ct-pt MACs (per
 * ciphertext), [3] bytes of scratch currently reserved, [4] kernel launches, [5] token blocks per group of the last
 * fesc_linear call, [6] passes of limb transforms outside fused conversions and inner products (two per transform); [7] zero. */
int fesc_ctx_counters(const fesc_ctx* ctx, uint64_t out[8]);
/*
 * Optional timing of kernel families with CUDA events recorded on the launching stream
 * (off by default; each timed launch costs two event records).  fesc_profile_enable(ctx, mask, n)
 * reserves n records and times the families whose bit is set in `mask` (0 = off); fesc_profile_read synchronises the device, returns
 * the summed milliseconds and record counts per family and clears the records.  Families:
 * 0 NTT/INTT, 1 ModUp conversion, 2 key inner product, 3 ModDown conversion and finish,
 * 4 automorphism gather, 5 BSGS accumulate, 6 rescale pointwise parts, 7 ct-pt MAC / tensor.
 * Launches beyond the reserved records are not timed.  Rings 2^10 .. 2^12: a key switch that would be one launch runs as its
 * steps while one of the families 0 to 3 is timed.
 */
int fesc_profile_enable(fesc_ctx* ctx, int mask, uint32_t max_records);
int fesc_profile_read(fesc_ctx* ctx, float ms[8], uint64_t records[8]);

/*
 * In-place forward / inverse negacyclic NTT of d_data (the evaluation representation of Sec. 2 "Fully Homomorphic
 * Encryption and CKKS": slot-wise products of ciphertexts and plaintexts are limb-wise products in this form) = [batch][n_limbs][N]; limb i is taken
 * modulo prime (first_limb + i) of the context's list (data primes, then special primes).
 * Input canonical; output canonical.  Forward output order: see "EVAL" above.
 */
int fesc_ntt(fesc_ctx* ctx, uint64_t* d_data, uint32_t batch, uint32_t first_limb,
             uint32_t n_limbs, void* stream);
int fesc_intt(fesc_ctx* ctx, uint64_t* d_data, uint32_t batch, uint32_t first_limb,
              uint32_t n_limbs, void* stream);

/*
 * ptmul + add (Table "CKKS primitives"): d_acc[b] += d_ct[b] (.) d_pt[b] on both polynomials,
 * EVAL form.  d_ct, d_acc: [batch][2][n_limbs][N]; d_pt: [batch][n_limbs][N] (pt_stride words
 * between consecutive plaintexts; 0 = the same plaintext for the whole batch).
 */
int fesc_ct_pt_mac(fesc_ctx* ctx, const uint64_t* d_ct, const uint64_t* d_pt, size_t pt_stride,
                   uint64_t* d_acc, uint32_t batch, uint32_t n_limbs, void* stream);

/*
 * rot / conj (Table "CKKS primitives"): the Galois automorphism FIRST, then a hybrid key switch
 * of the permuted c1:  (c0, c1) -> (sigma_g c0 + ks0, ks1).  Key switch: c1 to COEFF form;
 * per digit, uncorrected fast basis conversion to the other active moduli and the special
 * moduli (canonical representatives); inner product with the key; division by P with the
 * centred fast conversion of the special-limb residues.  d_in and d_out: [batch][2][n_limbs][N],
 * may not overlap.  The key must have been registered under key_id.
 */
int fesc_rotate(fesc_ctx* ctx, const uint64_t* d_in, uint64_t* d_out, uint32_t batch,
                uint32_t n_limbs, uint32_t key_id, void* stream);

/*
 * Hoisted rotations (a second, separately defined mode; not bit-identical to fesc_rotate): every input
 * ciphertext is decomposed ONCE (c1 to COEFF form, per-digit basis extension, NTT) and then rotated by each of
 * the n_keys registered keys: the automorphism is applied to the extended digits (a permutation in EVAL
 * form), followed by the inner product with that key and the division by P:
 *   out[k][b] = (sigma_g c0 + ks0, ks1),  ks = ModDown( sum_j sigma_g(d~_j) (.) key_{g,j} ).
 * The decrypted value is the same rotation; the residues differ from fesc_rotate because the conversion
 * overshoot is permuted instead of recomputed.  Saves 168 of 224 limb transforms per extra rotation at 24 limbs.
 * d_in [batch][2][n_limbs][N]; d_out [n_keys][batch][2][n_limbs][N], may not overlap d_in (FESC_EINVAL when they start
 * at the same address); key_ids: HOST array of n_keys ids.
 */
int fesc_rotate_hoisted(fesc_ctx* ctx, const uint64_t* d_in, uint64_t* d_out, uint32_t batch,
                        uint32_t n_limbs, const uint32_t* key_ids, uint32_t n_keys, void* stream);

/*
 * Rotate-and-add with one decomposition and one division by P (a separately defined mode; used by the radix-4
 * rotate-and-add chains of the scan-contract, where two doubling steps ct += rot(ct, d); ct += rot(ct, 2d) equal
 * ct + rot(ct, d) + rot(ct, 2d) + rot(ct, 3d)):
 *   out[b] = in[b] + sum_k rot_k(in[b]),
 *   out0 = c0 + sum_k sigma_k(c0) + ModDown( sum_k sum_j sigma_k(d~_j) (.) key_{k,j}[0] ),  out1 likewise with c1.
 * Same value as the sum of n_keys rotations (the division by P is additive up to its rounding); the residues
 * differ from summing fesc_rotate_hoisted outputs by at most n_keys units per coefficient.
 * d_in, d_out [batch][2][n_limbs][N], not overlapping; key_ids: HOST array of 1..8 registered key ids.
 */
int fesc_rotate_sum_hoisted(fesc_ctx* ctx, const uint64_t* d_in, uint64_t* d_out, uint32_t batch,
                            uint32_t n_limbs, const uint32_t* key_ids, uint32_t n_keys, void* stream);

/*
 * Rescale (Sec. 2 "Fully Homomorphic Encryption and CKKS": after a product the scale is divided out again and one
 * limb is consumed): rounded division by the last active prime, level n_limbs -> n_limbs-1:
 * c_i <- (c_i - [c_last]_centred) * q_last^-1 mod q_i.  d_in [batch][2][n_limbs][N],
 * d_out [batch][2][n_limbs-1][N]; may not overlap.  FESC_ELEVEL if n_limbs < 2.
 */
int fesc_rescale(fesc_ctx* ctx, const uint64_t* d_in, uint64_t* d_out, uint32_t batch,
                 uint32_t n_limbs, void* stream);

/*
 * The same rescale for callers that cannot allocate device memory (the paper has no counterpart of
 * this call; it exists for hosts of the library).  Who needs it: processes that have handed all of
 * HBM to another allocator under a fixed budget (a serving process that pre-partitions memory),
 * latency-critical loops that cannot afford the device-wide synchronisation an allocation implies,
 * and plug-in code whose host forbids allocator calls on its threads.  fesc_rescale takes its scratch (the last limb of every polynomial, batch*2*N
 * words) from the context arena, which may grow on first use; this variant keeps that scratch in a
 * fixed 4 MiB device array inside the library image (held by every GPU that loads the library until
 * the process exits) and calls no cudaMalloc, cudaFree or allocating library routine.
 *   - Limit: batch * 2 * N <= 524 288 words (4 ciphertexts at N = 2^16, 64 at N = 2^12); a larger
 *     batch is rejected with FESC_EINVAL and a message naming the limit: split it, or use fesc_rescale.
 *   - The first call on a device looks up the array's device address (cudaGetSymbolAddress, with that
 *     device current) and caches it per device ordinal.  With CUDA's lazy module loading that first call
 *     is also what loads the module and places the 4 MiB array on the device, so it can fail with
 *     FESC_ECUDA on a device whose memory has already been handed out: make it at initialisation, before
 *     the memory budget is given away and before any stream capture begins, and from one host thread
 *     (the cache is filled without locking; later calls only read it).
 *   - All calls share the one array.  Nothing in it has to start at zero (each call overwrites the
 *     rows it reads), but two calls that overlap on the GPU (different streams, or different
 *     contexts or threads) race on it: serialise them.
 * Arguments, layout and results are exactly those of fesc_rescale.
 */
int fesc_rescale_static(fesc_ctx* ctx, const uint64_t* d_in, uint64_t* d_out, uint32_t batch,
                        uint32_t n_limbs, void* stream);

/*
 * ctmul (Table "CKKS primitives") without the rescale: (d0,d1,d2) = (a0 b0, a0 b1 + a1 b0, a1 b1),
 * result (d0 + ks0, d1 + ks1) with ks = KeySwitch(d2, relinearisation key).  All operands
 * [batch][2][n_limbs][N]; d_out may alias neither input.
 */
int fesc_ct_ct_mul(fesc_ctx* ctx, const uint64_t* d_a, const uint64_t* d_b, uint64_t* d_out,
                   uint32_t batch, uint32_t n_limbs, void* stream);

/*
 * BSGS plaintext-weight projection Y = XW (App. "Projection Kernel Breakdown", real packing):
 * slot idx(r,c) = c*T + r of input ciphertext (tb, g) holds X[tb*T + r, g*C + c], C*T = N/2.
 *   acc_p = sum_g sum_{q<n1} rot(x^(tb,g), q*T) (.) D^(b)_{g,p,q}
 *   y^(tb,b) = sum_{p<n2} rot(acc_p, p*n1*T),  then rescale.
 * d_ct_in [token_blocks][in_blocks][2][n_limbs][N]
 * d_diags [out_blocks][n2][in_blocks][n1][n_limbs][N]   (encoded offline, EVAL form)
 * d_ct_out [token_blocks][out_blocks][2][n_limbs-1][N]
 * Galois keys: rotation by q*T under key id baby_key_base + q (q = 1..n1-1), rotation by
 * p*n1*T under giant_key_base + p (p = 1..n2-1); FESC_ENOKEY if one is missing.
 */
typedef struct fesc_bsgs_desc {
    uint32_t n1, n2;            /* baby / giant step counts, n1*n2 = C */
    uint32_t in_blocks;         /* ceil(d_in / C) */
    uint32_t out_blocks;        /* ceil(d_out / C) */
    uint32_t token_blocks;      /* ceil(tokens / T) */
    uint32_t n_limbs;           /* input level */
    uint32_t baby_key_base;
    uint32_t giant_key_base;
    uint32_t hoist;             /* 0: baby rotations by fesc_rotate; 1: by fesc_rotate_hoisted (other residues) */
    uint32_t defer;             /* 0: every giant rotation is a full fesc_rotate; 1: the inner products of the
                                   n2-1 giant steps are summed on the extended basis and divided by P once per
                                   output (same value, one rounding instead of n2-1; other residues when n2 > 2) */
    uint32_t packed;            /* 0: d_diags holds residues as laid out above; 1: d_diags is the byte-plane image
                                   written by fesc_linear_pack_diags (same results, bit for bit) */
    uint32_t diag_run_log2;     /* packed images only.  0: every coefficient of a diagonal has its own residue.  s > 0:
                                   the diagonals are PERIODIC plaintexts (slot vectors of period n / 2^s, as the
                                   token-major packing of the projection produces: slot r*C + c, feature shifts by the
                                   intra-segment shift Psi of App. "Projection Kernel Breakdown", masks folded into the
                                   diagonals); their evaluation form is constant on aligned runs of 2^s indices, the
                                   caller hands fesc_linear_pack_diags ONE word per run ([..][n_limbs][N >> s]) and the
                                   image is 2^s times smaller.  n1 and n2 then count the 2 n1' - 1 baby and 2 n2' - 1
                                   giant rotation amounts; the keys decide the amounts, as always. */
} fesc_bsgs_desc;
int fesc_linear(fesc_ctx* ctx, const uint64_t* d_ct_in, const uint64_t* d_diags,
                const fesc_bsgs_desc* desc, uint64_t* d_ct_out, void* stream);

/*
 * Packed diagonals.  The diagonals are weights: encoded once, used for every token.  fesc_linear_pack_diags rewrites
 * them, once, as the byte-plane operand tiles of the tensor-core accumulate (every residue below 2^56 cut into 7
 * bytes, terms in groups of 32, (b,p) pairs in tiles of 8, coefficients in tiles of 8; 7 bytes per residue instead
 * of 8), in the order one thread block streams them.  With desc->packed = 1 fesc_linear takes that image as d_diags
 * and forms the accumulators sum_{g,q} rot(x^(g), qT) (.) D_{g,p,q} as exact u8 x u8 -> s32 matrix products plus an
 * exact recombination: the output residues are identical to the unpacked call.
 *   fesc_linear_packed_bytes: size of the image for desc (n1, n2, in_blocks, out_blocks, n_limbs are read).
 *   fesc_linear_pack_diags: packs the (b,p) pairs [first, first + count) (pair index = b * n2 + p) from
 *     d_diags = [count][in_blocks][n1][n_limbs][N] residues (DEVICE) into their place inside d_packed (DEVICE, the
 *     whole image); `first` must be a multiple of 8 and only the last range may end inside a tile of 8, so the
 *     diagonals can be encoded and packed a few pairs at a time without ever holding all of them unpacked.
 * Needs N a multiple of 8, primes below 2^56 and at most 512 terms (in_blocks * n1); FESC_EINVAL otherwise.
 */
size_t fesc_linear_packed_bytes(const fesc_ctx* ctx, const fesc_bsgs_desc* desc);
int fesc_linear_pack_diags(fesc_ctx* ctx, const uint64_t* d_diags, const fesc_bsgs_desc* desc, uint32_t first,
                           uint32_t count, void* d_packed, void* stream);

/*
 * Real and imaginary slot parts of complex-packed ciphertexts (the projection pairs two real blocks in the real and
 * imaginary CKKS channels, App. "Projection Kernel Breakdown"), each DOUBLED, exact, same level:
 *   re2 = ct + conj(ct)  (slots 2 Re z),   im2 = -i (ct - conj(ct))  (slots 2 Im z),
 * conj = fesc_rotate under the conjugation key conj_key_id (registered with rot = FESC_CONJ).
 * With real weight diagonals a projection is linear over the complex slots, so fesc_linear on x^(2u) + i x^(2u+1)
 * followed by this split yields both real results for the cost of one projection plus one conjugation per output.
 * d_in, d_re2, d_im2 [batch][2][n_limbs][N], pairwise distinct; d_im2 may be NULL when only the real part is wanted
 * (input blocks paired with complex diagonals D^(2u) - i D^(2u+1): the real part of the accumulator is the result).
 */
int fesc_split_complex(fesc_ctx* ctx, const uint64_t* d_in, uint64_t* d_re2, uint64_t* d_im2, uint32_t batch,
                       uint32_t n_limbs, uint32_t conj_key_id, void* stream);

/*
 * Causal depthwise convolution (Sec. "Causal Depthwise Convolution", Eq. conv1d_depthwise) on the packing the
 * projection produces, slot idx(token, channel) = channel*T + token:
 *   eta_k[c] = b_c + sum_{r < d_conv} w_{c,r} q_{k-r}[c],  q_t = 0 for t < 0,
 * evaluated as  eta = bias + sum_r M_r (.) rho(q; -r) + sum_{r >= 1} M'_r (.) rho(q_prev; T - r),  then rescale:
 * M_r[c*T+k] = w_{c,r} for k >= r (0 elsewhere), M'_r[c*T+k] = w_{c,r} for k < r (the first r tokens of a block read
 * the last tokens of the previous token block; absent for the first block).  The 2(d_conv-1) rotations of one
 * ciphertext are hoisted rotations (fesc_rotate_hoisted).
 * d_ct_in  [token_blocks][blocks][2][n_limbs][N]
 * d_masks  [blocks][2*d_conv-1][n_limbs][N]   M_0..M_{d_conv-1}, M'_1..M'_{d_conv-1}, EVAL form, encoded offline
 * d_bias   [blocks][n_limbs][N]               encoded at the scale of the products (input scale x mask scale)
 * d_ct_out [token_blocks][blocks][2][n_limbs-1][N]
 * Galois keys: rotation by -r under key id key_base + r, rotation by T - r under key_base + d_conv + r (r = 1..d_conv-1;
 * the second family only when token_blocks > 1); FESC_ENOKEY if one is missing.  d_conv <= 8.
 */
typedef struct fesc_conv_desc {
    uint32_t d_conv;        /* taps */
    uint32_t T;             /* tokens per segment (slots per channel) */
    uint32_t blocks;        /* channel blocks (ciphertexts per token block) */
    uint32_t token_blocks;
    uint32_t n_limbs;       /* input level */
    uint32_t key_base;
} fesc_conv_desc;
int fesc_conv(fesc_ctx* ctx, const uint64_t* d_ct_in, const uint64_t* d_masks, const uint64_t* d_bias,
              const fesc_conv_desc* desc, uint64_t* d_ct_out, void* stream);

/*
 * The CKKS steps around the NeRMS protocol (Alg. "one Block"), on the same packing slot = channel*T + token.
 *
 * fesc_norm_square:  u = y~ (.) y~  (the squares the protocol turns into one inverse RMS per token): ciphertext product,
 * relinearisation, rescale.  d_y [batch][2][n_limbs][N] -> d_out [batch][2][n_limbs-1][N].  n_limbs >= 2.
 *
 * fesc_norm_scale:  y^ = gamma_RMS (.) (y~ (.) br(s_RMS))  (the input of HEOutProj).
 * d_y     [token_blocks][blocks][2][n_limbs][N]  gated scan output of every (token block, channel block)
 * d_s     [token_blocks][2][n_limbs][N]          slot k < T = the factor of token k, every other slot 0
 * d_gamma [blocks][n_limbs-1][N]                 plaintexts, EVAL form, slot c*T + k = weight of channel c of the block
 * d_out   [token_blocks][blocks][2][n_limbs-2][N]
 * br(s): log2(n/T) rotate-right-and-add steps f += rot(f, -(T << b)), b = 0, 1, ... (shared by the channel blocks of a
 * token block); then y~ (.) br(s) relinearised and rescaled, the plaintext product with gamma, and a second rescale.
 * Galois keys: the rotation by -(T << b) under key id key_base + b; FESC_ENOKEY if one is missing.  T a power of two
 * that divides n; n_limbs >= 3 (FESC_ELEVEL otherwise).
 */
typedef struct fesc_norm_desc {
    uint32_t T;             /* tokens per segment (slots per channel) */
    uint32_t blocks;        /* channel blocks (ciphertexts per token block) */
    uint32_t token_blocks;
    uint32_t n_limbs;       /* input level */
    uint32_t key_base;
} fesc_norm_desc;
int fesc_norm_square(fesc_ctx* ctx, const uint64_t* d_y, uint64_t* d_out, uint32_t batch, uint32_t n_limbs, void* stream);
int fesc_norm_scale(fesc_ctx* ctx, const uint64_t* d_y, const uint64_t* d_s, const uint64_t* d_gamma,
                    const fesc_norm_desc* desc, uint64_t* d_out, void* stream);

/*
 * Factorized scan-contract (Sec. 5.4, Eqs. fesc_recurrence / fesc_contract):
 *   h_k = br(a_k) (.) h_{k-1} + x_k (x) B_k,  h_0 = 0,   m_k = Sigma_{d_s}(h_k (.) br(C_k)),
 * x_k in R^{H x P}, a_k in R^H, B_k, C_k in R^{d_s} (one group).  Only the compact factors enter and
 * only m leaves; states exist per (token block, state chunk) inside the call.
 *
 * Geometry (powers of two): n = N/2 slots = c_state * stride, stride >= d_s (0 selects max(d_s, B_blk));
 * chunk kappa owns channels [kappa*c_state, (kappa+1)*c_state), K_s = H*P / c_state;
 * hpc = c_state / P heads per chunk, each a region of R = n / hpc slots; K_blk = ceil(L / B_blk).
 * A block is cut into segs = max(1, B_blk/stride) token segments of Bt = B_blk/segs tokens, with one x, a and
 * output ciphertext per segment: stride >= B_blk is one segment (with stride = 256 > d_s = 128 half of the state
 * slots stay idle, the paper's s_state = n/2); stride = d_s < B_blk uses every slot (s_state = n) and needs half as
 * many chunks for the same channels.  Requires B_blk*d_s <= n and Bt*P <= R.
 * Inputs at level n_limbs = l0, t = token within block j, t = seg*Bt + t':
 *   d_x [K_blk][K_s][segs][2][l0][N]: slot e'*stride + t' = x_{j*B_blk+t}[kappa*c_state + e']
 *   d_a [K_blk][K_s][segs][2][l0][N]: slot hh*R + t'*P    = a_{j*B_blk+t}[kappa*hpc + hh], other slots 0
 *   d_B, d_C [K_blk][2][l0][N]:       slot t*d_s + i      = B_{j*B_blk+t}[i], C_{j*B_blk+t}[i]
 * Output d_m_out [K_blk][K_s][segs][2][l_out][N]: slot e'*stride + t' = m_{j*B_blk+t}[kappa*c_state + e'].
 * (Token offsets t' of x, a and the output placement use the two digits t' = t_lo + min(16,Bt) t_hi.)
 *
 * Dataflow (Eq. compact_affine_compose, Eq. hescan-contract-output, Eq. resident-block-schedule with
 * serialized carries, Brent-Kung network of App. "Prefix-Network Selection", paired reduction of App.
 * "Complex-Packed Reduction Accounting"): per block, br(B_t), br(C_t) by rotation by t*d_s (two-digit
 * offsets t = t_lo + 16 t_hi), mask, log2(c_state) rotate-right-and-add steps of stride*2^b; per chunk,
 * br(x_t) (rotation by t, mask, log2(d_s) steps of 2^b), br(a_t) (pre-fill log2(P) steps, rotation by
 * t*P, mask, log2(R/P) steps of P*2^b), leaves (br a_t, br x_t (.) br B_t); up-sweep stages s = 1..log2 B
 * at every position k multiple of 2^s, down-sweep stages s = log2 B - 1..1 at every k multiple of 2^s
 * with k + 2^(s-1) < B (1-based), each node (p_R p_L, p_R s_L + s_R); carry g_{j+1} = p_S g_j + s_S;
 * state = p g_j + s; contraction with br(C_t); chunks (2l, 2l+1) reduced together as v + i v' by
 * log2(d_s) rotate-left-and-add steps and one conjugation; output mask; rotation right by t; sum.
 * Level schedule (logB = log2 B_blk): masked factors l0-1 (br(C_t) is brought down to linj-1 after its mask and
 * filled there); leaves l1 = l0-2; up-sweep stage s -> l1-s; lS = l1-logB;
 * down-sweep stage number d works at lS-(d-1); carry before block j >= 1 at lS-(j-1); injection at
 * linj = l1-2logB+1; contraction at linj-1; reduction at linj-2; output l_out = linj-3.  An operand at
 * a higher level is brought down by: keep its first dst+1 limbs, multiply by the integer
 * adj[src*(l0+1)+dst], rescale.  FESC_ELEVEL if l_out < 1 or the carries would pass linj.
 *
 * Constants come from the caller (the library does no floating point): plaintext masks in EVAL form
 * (DEVICE): mask_x (slots = 0 mod stride), mask_b (slots [0,d_s)), mask_a (slots [hh*R, hh*R+P)) at
 * level l0, mask_out (slots = 0 mod stride) at level linj-2; HOST tables adj_s, adj_p of (l0+1)^2
 * integers for state-like and multiplicand ciphertexts.  Galois keys: rotation by r slots must be
 * registered under key_base + (r mod n), conjugation under key_base + n; FESC_ENOKEY otherwise.
 * Scratch grows to the peak of one (block, chunk) working set.
 */
typedef struct fesc_scan_desc {
    uint32_t L, H, P, d_s, B_blk;
    uint32_t stride;        /* 0 = max(d_s, B_blk) */
    uint32_t n_limbs;       /* l0 */
    uint32_t key_base;
    uint32_t hoist;         /* 0: every rotation is a fesc_rotate.  1 (a separately defined mode, other residues, same
                               values): rotate-and-add chains take two doubling steps at once through
                               fesc_rotate_sum_hoisted (keys for 3 * unit * 2^b are needed as well, b even), and the
                               low digit of the two-digit token offsets uses fesc_rotate_hoisted */
    uint32_t network;       /* prefix network over the positions of a block (App. "Prefix-Network Selection"):
                               FESC_NET_BRENT_KUNG (0, the schedule above); FESC_NET_KOGGE_STONE: stage s = 1..logB, every
                               position k > 2^(s-1) (1-based) takes t_{k-2^(s-1)} o t_k of stage s-1; FESC_NET_SKLANSKY:
                               stage s, the upper half of every aligned block of 2^s takes (last of the lower half) o t_k.
                               Both work at l1-(s-1) -> l1-s, finish every prefix at lS and have no down-sweep:
                               linj = lS - max(K_blk-2, 0), the other levels follow from linj as above. */
    uint32_t group;         /* 0: br(x_t), br(a_t) are built token by token (above).  G >= 2 (a power of two, at most 16,
                               the tokens of a segment and d_s; a separately defined mode, other residues, same
                               values): groups of G consecutive
                               tokens are extracted (rotation by G*u resp. G*P*u), masked (d_mask_xg, d_mask_ag) and
                               filled once (log2(d_s/G) steps of G*2^b, log2(R/(G*P)) steps of G*P*2^b); the group
                               ciphertext is rotated once by +-unit .. +-(G-1)*unit (unit 1 for x, P for a; hoisted
                               rotations when hoist = 1) and the token of class c = t mod G is
                               rescale(sum_{j<G} mask2[j] (.) rot(group, (c - j)*unit)) with the class masks d_mask_x2,
                               d_mask_a2; br(a_t) is then brought to l1.  br(B_t) is built the same way (groups =
                               G*d_s consecutive slots, rotation by G*d_s*u, d_mask_bg, log2(n/(G*d_s)) steps of
                               G*d_s*2^b, class shifts of d_s slots, d_mask_b2) and lands at l0-2.  The class masks
                               cost a level: leaves at l1 = l0-3, every later level one lower than above. */
    uint32_t plain;         /* 0: selective scan, a, B, C encrypted (above).  1: invariant families (App. "Invariant
                               Families", "Shared HEScan Kernel Backend"; S4D, S5, LRU): the decay abar[i] per state
                               coordinate, the input factor Bbar[i] and the output factor Cbar[i] are plaintexts that do
                               not depend on the token, only x is encrypted:
                                 h_k[e,i] = abar[i] h_{k-1}[e,i] + x_k[e] Bbar[i],   m_k[e] = sum_i h_k[e,i] Cbar[i].
                               d_a, d_B, d_C are ignored (may be NULL).  The packet has no decay component: a composition
                               over a span of m tokens is s <- abar^m (.) s_L + s_R, ONE ct-pt product; no ciphertext
                               product and no relinearisation anywhere.  Same layouts, br(x_t) build (hoist, group), level
                               schedule, carries and reduction; Brent-Kung network only.  The plaintexts come from the
                               caller in fesc_scan_consts (d_pt_*), each the slot pattern e'*stride + i -> v[i] (0 for
                               i >= d_s) in EVAL form at the multiplicand scale of the level where it is used. */
} fesc_scan_desc;
enum { FESC_NET_BRENT_KUNG = 0, FESC_NET_KOGGE_STONE = 1, FESC_NET_SKLANSKY = 2 };
typedef struct fesc_scan_consts {
    const uint64_t* d_mask_x;    /* device [l0][N] */
    const uint64_t* d_mask_b;    /* device [l0][N] */
    const uint64_t* d_mask_a;    /* device [l0][N] */
    const uint64_t* d_mask_out;  /* device [linj-2][N] */
    const uint64_t* adj_s;       /* host [(l0+1)*(l0+1)] */
    const uint64_t* adj_p;       /* host [(l0+1)*(l0+1)] */
    /* grouped leaf build only (desc.group = G), else NULL: */
    const uint64_t* d_mask_xg;   /* device [l0][N]: slots with (slot mod stride) < G */
    const uint64_t* d_mask_ag;   /* device [l0][N]: slots with (slot mod R) < G*P */
    const uint64_t* d_mask_x2;   /* device [G][l0-1][N]: class c = slots with (slot mod stride) < d_s and = c mod G */
    const uint64_t* d_mask_a2;   /* device [G][l0-1][N]: class c = slots with floor((slot mod R) / P) = c mod G */
    const uint64_t* d_mask_bg;   /* device [l0][N]: slots below G*d_s */
    const uint64_t* d_mask_b2;   /* device [G][l0-1][N]: class c = slots with floor(slot / d_s) = c mod G */
    /* invariant-family mode only (desc.plain = 1), else NULL; tables with one level per row use a row pitch of l0*N words: */
    const uint64_t* d_pt_b;      /* device [lx][N], lx = level of br(x_t) (l0-1; l0-2 with group): Bbar */
    const uint64_t* d_pt_c;      /* device [linj-1][N]: Cbar */
    const uint64_t* d_pt_up;     /* device [logB][l0][N]: row s-1 = abar^(2^(s-1)) at level l1-(s-1) (up-sweep stage s) */
    const uint64_t* d_pt_down;   /* device [logB-1][l0][N]: row d-1 = abar^(2^(logB-d-1)) at level lS-(d-1) (down-sweep stage number d) */
    const uint64_t* d_pt_carry;  /* device [K_blk][l0][N]: row j (1 <= j <= K_blk-2) = abar^B_blk at level lS-(j-1) */
    const uint64_t* d_pt_inj;    /* device [B_blk][linj][N]: row t = abar^(t+1) at level linj (NULL when K_blk = 1) */
} fesc_scan_consts;
int fesc_scan_contract(fesc_ctx* ctx, const uint64_t* d_x, const uint64_t* d_a, const uint64_t* d_B,
                       const uint64_t* d_C, const fesc_scan_desc* desc, const fesc_scan_consts* consts,
                       uint64_t* d_m_out, void* stream);

#ifdef __cplusplus
}
#endif
#endif /* FESC_H */

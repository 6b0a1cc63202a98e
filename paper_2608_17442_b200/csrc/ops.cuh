// Internal interfaces between the ciphertext-operation translation units.
#pragma once
#include "common.cuh"

// Scratch of one key-switch chunk (all [chunk][...][N] words):
//   dcoef [level]            the polynomial being switched, transformed to COEFF in place
//   ext   [beta][level+K]    converted digits; the rows of a digit's own limbs hold the polynomial itself (EVAL);
//                            n_ext such buffers in a row when several polynomials are switched before one sum
//   acc   [2][level+K]       inner-product accumulators
//   u     [2][level]         converted special-limb part
struct KsScratch {
    u64 *dcoef, *ext, *acc, *u;
};
// Several sources can be summed in one pass: source s contributes sum_j dt_j(ext_s)[pi_{g_s}(t)] * key_s[j].  The giant
// steps of a projection (different converted polynomials, different keys, one sum) and the rotate-and-add chains (one
// converted polynomial read through several Galois permutations, one key each) then read and write the accumulators
// once instead of once per key, and the later reads of a shared source hit L2.
#define INNER_MAX_SRC KS_MAX_KEYS
struct InnerSrc {
    const u64* ext;   // [batch][beta][level+K][N]
    const u64* key;   // [beta][2][n_q+K][N]
    u64 g;            // Galois element the digits are read through (0: none)
};
struct InnerSrcs {
    InnerSrc s[INNER_MAX_SRC];
    uint32_t n;
};

// How a key-switch pass is cut and its scratch in polynomials: `src` are decomposed at a time (dcoef), `ext` converted ones are kept,
// `acc` accumulators (and converted special parts) exist side by side.
struct KsCut {
    uint32_t nb, keys;          // ciphertexts and keys per pass
    uint32_t src, ext, acc;
};
// one key per call, or several plain rotations of the same few ciphertexts: keys share a pass until it has 16 polynomials
KsCut ks_cut_rotate(const fesc_ctx* ctx, uint32_t batch, uint32_t n_keys = 1);
// hoisted rotations: one decomposition, the keys of a pass share one reading of the converted digits and one division launch
KsCut ks_cut_hoisted(const fesc_ctx* ctx, uint32_t batch, uint32_t n_keys);
// deferred giant-step sum over n_terms - 1 rotated terms
KsCut ks_cut_giant(const fesc_ctx* ctx, uint32_t batch, uint32_t n_terms);
size_t ks_scratch_words(const fesc_ctx* ctx, uint32_t level, const KsCut& cut);
KsScratch ks_scratch_carve(const fesc_ctx* ctx, u64* base, uint32_t level, const KsCut& cut);
int rotate_internal(fesc_ctx* ctx, const u64* in, size_t in_stride, u64* out, size_t out_stride, uint32_t batch,
                    uint32_t level, uint32_t key_id, u64* scratch, cudaStream_t st, int accumulate);
int rotate_hoisted_internal(fesc_ctx* ctx, const u64* in, size_t in_stride, u64* out, size_t out_stride,
                            size_t key_stride, uint32_t batch, uint32_t level, const uint32_t* key_ids, uint32_t n_keys,
                            u64* scratch, cudaStream_t st);
int rotate_sum_hoisted_internal(fesc_ctx* ctx, const u64* in, size_t in_stride, u64* out, size_t out_stride,
                                uint32_t batch, uint32_t level, const uint32_t* key_ids, uint32_t n_keys, u64* scratch,
                                cudaStream_t st);
// Plain rotations of the same kind of ciphertexts by n_keys keys: rotation of ciphertext b (at in + k * in_key_stride + b * in_stride) by
// key k to out + k * out_key_stride + b * out_stride; accumulate: added to what is there.
int rotate_multi_internal(fesc_ctx* ctx, const u64* in, size_t in_stride, size_t in_key_stride, u64* out, size_t out_stride,
                          size_t out_key_stride, uint32_t batch, uint32_t level, const uint32_t* key_ids, uint32_t n_keys, u64* scratch,
                          cudaStream_t st, int accumulate);
int giant_sum_deferred_internal(fesc_ctx* ctx, u64* acc, uint32_t n_terms, size_t ct_words, uint32_t batch,
                                uint32_t level, uint32_t key_base, u64* scratch, cudaStream_t st);
// out[b] = sum_j src_j[b] (.) pt_j[b] (+ add[b] on the first polynomial), at most 16 terms
struct MaskedSum {
    const u64 *src[16], *pt[16];
    uint32_t n;
};
int masked_sum(fesc_ctx* ctx, const MaskedSum& s, size_t src_stride, size_t pt_stride, const u64* add, size_t add_stride, u64* out,
               size_t out_stride, uint32_t batch, uint32_t level, cudaStream_t st);
// What the rescale takes beyond a contiguous batch, where rescale_fused holds: polynomials stored with more limbs than `level`, a product
// (by plaintexts at pt + b * pt_stride, or by an integer) that is formed on the way, results with a stride (then `rows` holds the
// batch * 2 * (level - 1) rows of the transform).
struct RescaleView {
    uint32_t in_rows = 0;           // limbs per stored polynomial; 0: level
    const u64* pt = nullptr;        // [level][N]
    size_t pt_stride = 0;
    u64 mul = 0;                    // 0: none
    size_t out_stride = 0;          // 0: contiguous
    u64* rows = nullptr;
};
bool rescale_fused(const fesc_ctx* ctx, uint32_t level);
int rescale_internal(fesc_ctx* ctx, const u64* in, size_t in_stride, u64* out, uint32_t batch, uint32_t level,
                     u64* scratch, cudaStream_t st, const RescaleView& view = RescaleView());
int ctmul_internal(fesc_ctx* ctx, const u64* a, size_t a_stride, const u64* b, size_t b_stride, u64* out,
                   size_t out_stride, uint32_t batch, uint32_t level, u64* scratch, cudaStream_t st);

// ---------------------------------------------------------------------------------------
// Byte-plane products on the tensor cores (BSGS accumulate): u8 x u8 -> s32 mma.sync m16n8k32 and the recombination
// of the 7 x 7 byte-plane sums of one output.
// ---------------------------------------------------------------------------------------
#ifdef __CUDACC__
__device__ __forceinline__ void imma_u8(int (&d)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0,
                                        uint32_t b1) {
    asm volatile("mma.sync.aligned.m16n8k32.row.col.s32.u8.u8.s32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
                 : "+r"(d[0]), "+r"(d[1]), "+r"(d[2]), "+r"(d[3])
                 : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}
// the same product with zero addends (first k-step of a tile).  z0..z3 are four registers that hold zero and are kept
// opaque to the optimiser, so that they stay one fixed operand quad instead of being rebuilt before every instruction.
__device__ __forceinline__ void imma_u8_zero(int (&d)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0,
                                             uint32_t b1, int z0, int z1, int z2, int z3) {
    asm volatile("mma.sync.aligned.m16n8k32.row.col.s32.u8.u8.s32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%10,%11,%12,%13};"
                 : "=r"(d[0]), "=r"(d[1]), "=r"(d[2]), "=r"(d[3])
                 : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1), "r"(z0), "r"(z1), "r"(z2), "r"(z3));
}
// d[k] = (byte k of w0) | (byte k of w1) << 8 | (byte k of w2) << 16 | (byte k of w3) << 24, k = 0..6
__device__ __forceinline__ void byte_planes4(u64 w0, u64 w1, u64 w2, u64 w3, uint32_t (&d)[7]) {
    const uint32_t l0 = (uint32_t)w0, l1 = (uint32_t)w1, l2 = (uint32_t)w2, l3 = (uint32_t)w3;
    const uint32_t h0 = (uint32_t)(w0 >> 32), h1 = (uint32_t)(w1 >> 32), h2 = (uint32_t)(w2 >> 32), h3 = (uint32_t)(w3 >> 32);
    const uint32_t t0 = __byte_perm(l0, l1, 0x5140), t1 = __byte_perm(l2, l3, 0x5140);
    const uint32_t t2 = __byte_perm(l0, l1, 0x7362), t3 = __byte_perm(l2, l3, 0x7362);
    d[0] = __byte_perm(t0, t1, 0x5410);
    d[1] = __byte_perm(t0, t1, 0x7632);
    d[2] = __byte_perm(t2, t3, 0x5410);
    d[3] = __byte_perm(t2, t3, 0x7632);
    const uint32_t u0 = __byte_perm(h0, h1, 0x5140), u1 = __byte_perm(h2, h3, 0x5140);
    const uint32_t u2 = __byte_perm(h0, h1, 0x7362), u3 = __byte_perm(h2, h3, 0x7362);
    d[4] = __byte_perm(u0, u1, 0x5410);
    d[5] = __byte_perm(u0, u1, 0x7632);
    d[6] = __byte_perm(u2, u3, 0x5410);
}
// Recombination.  d[m][j][r]: accumulators of m-tile m (byte planes 2m, 2m+1 of the diagonal side), n-tile j (byte plane
// j of the input side); registers r = 0,1 belong to plane 2m and r = 2,3 to plane 2m+1, r & 1 = sel picks the polynomial.
// E_d = sum_{k+j=d} D[k][j] (13 values; below 2^28 for at most 512 terms), four of them are packed exactly into one
// integer T_m < 2^52, and S = T_0 + T_1 2^32 + T_2 2^64 + T_3 2^96 is reduced modulo q: with exact FP64 products for
// primes below 2^50 (|fp_reduce| <= q/2 and every lazy product within 2q, so the sum stays below 6.5 q < 2^53), as a
// 128-bit integer otherwise.  c32, c64, c96 = 2^32, 2^64, 2^96 mod q (FP path only).
template <bool FP>
__device__ __forceinline__ u64 imma_reduce(const uint32_t (&e)[13], const PrimeConst& pc, double c32, double c64, double c96) {
    const u64 w0 = e[0] + ((u64)e[1] << 8) + ((u64)e[2] << 16) + ((u64)e[3] << 24);
    const u64 w1 = e[4] + ((u64)e[5] << 8) + ((u64)e[6] << 16) + ((u64)e[7] << 24);
    const u64 w2 = e[8] + ((u64)e[9] << 8) + ((u64)e[10] << 16) + ((u64)e[11] << 24);
    if (FP) {
        const double q = pc.qd, qinv = pc.qinvd;
        const double r = fp_reduce(fp_from_u64(w0), q, qinv) + fp_modmul(fp_from_u64(w1), c32, q, qinv) +
                         fp_modmul(fp_from_u64(w2), c64, q, qinv) + fp_modmul(fp_from_u64((u64)e[12]), c96, q, qinv);
        return fp_store(r, q, qinv);
    }
    const u128 S = (u128)w0 + ((u128)w1 << 32) + ((u128)w2 << 64) + ((u128)e[12] << 96);
    return reduce128((u64)(S >> 64), (u64)S, pc);
}
template <bool FP>
__device__ __forceinline__ u64 imma_recombine(const int (&d)[4][7][4], int sel, const PrimeConst& pc, double c32, double c64,
                                              double c96) {
    uint32_t e[13];
#pragma unroll
    for (int x = 0; x < 13; x++) e[x] = 0;
#pragma unroll
    for (int k = 0; k < 7; k++)
#pragma unroll
        for (int j = 0; j < 7; j++) e[k + j] += (uint32_t)d[k >> 1][j][(k & 1) * 2 + sel];
    return imma_reduce<FP>(e, pc, c32, c64, c96);
}
#endif

// basis conversions on the tensor cores (bconv.cu)
bool bconv_supported(const fesc_ctx* ctx, uint32_t level);
void moddown_conv_imma_launch(fesc_ctx* ctx, const u64* acc, u64* u, uint32_t level, uint32_t batch, int out_double, cudaStream_t st);

// ModUp fused with the first eight stages of the forward transform (N = 2^16, modup16.cu): y = the COEFF rows times
// (Q_j/q_a)^-1
bool modup16_supported(const fesc_ctx* ctx, uint32_t level);
// the same for the division by P: the special rows of acc hold COEFF residues times (P/p_k)^-1
bool moddown16_supported(const fesc_ctx* ctx, uint32_t level);
bool moddown16_open(const fesc_ctx* ctx, uint32_t level);      // the special rows arrive without the last pass of their inverse transform
int moddown16_cols_launch(fesc_ctx* ctx, const u64* acc, u64* u, uint32_t level, uint32_t polys, cudaStream_t st);
int modup16_cols_launch(fesc_ctx* ctx, const u64* y, u64* ext, uint32_t level, uint32_t batch, cudaStream_t st);

// rows on primes below 2^50: last pass of the forward transform of the converted digits and key inner product in one kernel (inner16.cu)
// inv_special: the special rows are left after the first pass of their inverse transform
int rows_inner_launch(fesc_ctx* ctx, const InnerSrcs& S, u64* acc, uint32_t level, uint32_t batch, int accumulate, bool separate, bool inv_special,
                      cudaStream_t st);

// rings N = 2^10 .. 2^12 (small.cu): the steps of a key switch and of a rescale, one row per CTA.  small_inner with `last` leaves the
// special rows of acc in the form small_moddown takes.
bool small_ring(const fesc_ctx* ctx);
int small_decompose(fesc_ctx* ctx, const KsScratch& ws, const u64* src, size_t src_stride, bool keep_own, u64 g, uint32_t level, uint32_t batch,
                    cudaStream_t st);
int small_inner(fesc_ctx* ctx, const KsScratch& ws, const InnerSrcs& S, uint32_t level, uint32_t batch, cudaStream_t st, int accumulate, int last);
int small_moddown(fesc_ctx* ctx, const KsScratch& ws, uint32_t level, uint32_t batch, u64* out, size_t out_stride, int add_mask, cudaStream_t st,
                  const u64* rot_src, size_t rot_stride, u64 g);
// a whole key switch with one key in one launch where the call is small enough (false: the steps above have to be used)
bool small_switch(fesc_ctx* ctx, const KsScratch& ws, const u64* src, size_t src_stride, bool keep_own, u64 g, const u64* key, uint32_t level, uint32_t batch,
                  u64* out, size_t out_stride, int add_mask, cudaStream_t st, const u64* rot_src, size_t rot_stride, int& rc);
int small_rescale(fesc_ctx* ctx, const u64* in, size_t in_stride, u64* out, size_t out_stride, uint32_t batch, uint32_t level, u64* r, cudaStream_t st);

// packed-operand BSGS accumulate (packed.cu)
size_t bsgs_packed_bytes(uint32_t N, uint32_t level, uint32_t rows, uint32_t terms);
bool bsgs_packed_supported(const fesc_ctx* ctx, uint32_t level, uint32_t terms, uint32_t dshift);
int bsgs_pack_inputs(fesc_ctx* ctx, const u64* rot, uint8_t* xpk, uint32_t level, uint32_t tbs, uint32_t terms, bool cores, cudaStream_t st);
int bsgs_accumulate_packed(fesc_ctx* ctx, const uint8_t* xpk, const uint8_t* dpk, u64* acc, uint32_t level, uint32_t tbs,
                           uint32_t terms, uint32_t bp_count, bool fp, uint32_t dshift, cudaStream_t st);
// the same for periodic diagonals (packed_tc.cu); its inputs are packed with `cores`
bool bsgs_periodic_supported(uint32_t terms, uint32_t bp_count, uint32_t dshift);
int bsgs_accumulate_periodic(fesc_ctx* ctx, const uint8_t* xpk, const uint8_t* dpk, u64* acc, uint32_t level, uint32_t tbs, uint32_t terms,
                             uint32_t bp_count, bool fp, uint32_t dshift, cudaStream_t st);

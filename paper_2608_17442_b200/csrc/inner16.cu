// Key inner product fused with the last pass of the forward transform (N = 2^16, rows on primes below 2^50):
//   acc[b][p][t] = sum_s sum_j NTT(ext_s[b][j][t]) * key_s[j][p][t]
// for key switches whose converted digits serve one key only (rotations, relinearisation, giant-step sums; hoisted rotations keep
// the transformed digits for several keys).  The transformed rows are never stored: 75 MB written and 88 MB read per ciphertext at
// 24 limbs.
//
// Measured on 128 rotations at 24 limbs (batches of 16): 5.84 ms and 2.7 ms less in the transforms, against 3.45 ms for the inner
// product on stored digits; FP64 pipe 55 %, the rest is latency at 16 warps per SM.  Staging the next digit's points through shared
// memory with asynchronous copies was slower (9.2 ms): it takes the L1 from the key words and twiddles that the warps share.
//
// The special rows arrive transformed and are multiplied by the last CTAs of the same launch: their products and loads run beside the
// data rows' arithmetic and fill its last wave (5.36 + 0.98 ms in two launches, 5.84 ms in one; first instead of last 6.02).  Two warps per 512 points with
// half the digits each, for single ciphertexts: 103 us against 86.
//
// A warp owns 512 points of one row of one ciphertext.  It runs rounds C and D of every digit in turn (the digit that holds the row
// itself needs no transform), multiplies with the two key words of each point and keeps both sums in registers; 128 registers, 16
// warps per SM.  The four warps of a CTA are four ciphertexts on the same points, so that the key words come from L1 after the first.
#define FESC_DBG_FILE 14   // file id in the sites a debug build reports
#include "ntt16.cuh"
#include "ops.cuh"

#define RI_WARPS 4
// The special rows (integers, stored transformed): 512 points of one ciphertext per warp, four points of a lane at a time.
__device__ __forceinline__ void int_rows(const InnerSrcs& S, uint32_t s0, uint32_t s1, u64* o0, u64* o1, const PrimeConst& pc, size_t x_at, size_t x_step,
                                         size_t key_at, size_t key_step, uint32_t beta, int accumulate) {
#pragma unroll 1
    for (int k = 0; k < 512; k += 128) {
        acc128 a[8] = {};
        uint32_t n = 0;
        for (uint32_t s = s0; s < s1; s++) {
            const u64 *x = S.s[s].ext + x_at + k, *key = S.s[s].key + key_at + k;
#pragma unroll 2
            for (uint32_t j = 0; j < beta; j++, x += x_step, key += 2 * key_step) {
#pragma unroll
                for (int h = 0; h < 2; h++) {
                    const ulonglong2 v = *reinterpret_cast<const ulonglong2*>(x + 64 * h);
                    const ulonglong2 w0 = __ldg(reinterpret_cast<const ulonglong2*>(key + 64 * h));
                    const ulonglong2 w1 = __ldg(reinterpret_cast<const ulonglong2*>(key + key_step + 64 * h));
                    mac128(a[4 * h], v.x, w0.x);
                    mac128(a[4 * h + 1], v.y, w0.y);
                    mac128(a[4 * h + 2], v.x, w1.x);
                    mac128(a[4 * h + 3], v.y, w1.y);
                }
                if ((++n & 7) == 0) {               // eight products below 2^124 fit 128 bits
#pragma unroll
                    for (int i = 0; i < 8; i++) a[i] = acc128{reduce128(a[i].hi, a[i].lo, pc), 0};
                }
            }
        }
#pragma unroll
        for (int i = 0; i < 4; i++) {
            ulonglong2* o = reinterpret_cast<ulonglong2*>((i & 1 ? o1 : o0) + k + 64 * (i >> 1));
            ulonglong2 r = make_ulonglong2(reduce128(a[2 * i].hi, a[2 * i].lo, pc), reduce128(a[2 * i + 1].hi, a[2 * i + 1].lo, pc));
            if (accumulate) {
                const ulonglong2 v = *o;
                r.x = addmod(r.x, v.x, pc.q), r.y = addmod(r.y, v.y, pc.q);
            }
            *o = r;
        }
    }
}

__global__ void __launch_bounds__(32 * RI_WARPS, 4)
    k_rows_inner(InnerSrcs S, u64* acc, const double* __restrict__ twf, const PrimeConst* __restrict__ pcs, uint32_t level, uint32_t n_q,
                 uint32_t K, uint32_t alpha, uint32_t beta, uint32_t batch, int accumulate, int sep) {
    pdl_begin();
    __shared__ __align__(16) u64 sm_all[RI_WARPS * ROW_SMEM];
    const uint32_t lane = threadIdx.x & 31, warp = threadIdx.x >> 5, id = blockIdx.x * RI_WARPS + warp;
    const uint32_t blk = id / batch, b = id - blk * batch, t = blockIdx.y, rows = level + K, np = n_q + K;
    const uint32_t pt = t < level ? t : n_q + (t - level), own = t / alpha;
    if (blk >= 128) return;                             // warp barriers only
    const uint32_t s0 = sep ? blockIdx.z : 0, s1 = sep ? s0 + 1 : S.n;
    acc += (size_t)s0 * batch * 2 * rows * N16;         // separate sources have their own accumulators
    u64* o0 = acc + ((size_t)b * 2 * rows + t) * N16 + blk * 512 + 2 * lane;
    u64* o1 = o0 + (size_t)rows * N16;
    bool ok = DBG_REGION(o0 - 2 * lane, 512 * sizeof(u64)) && DBG_REGION(o1 - 2 * lane, 512 * sizeof(u64));
    for (uint32_t s = s0; s < s1; s++)
        for (uint32_t j = 0; j < beta; j++)
            ok = ok && DBG_REGION(S.s[s].ext + (((size_t)b * beta + j) * rows + t) * N16 + blk * 512, 512 * sizeof(u64)) &&
                 DBG_REGION(S.s[s].key + ((size_t)(2 * j) * np + pt) * N16, N16 * sizeof(u64)) &&
                 DBG_REGION(S.s[s].key + ((size_t)(2 * j + 1) * np + pt) * N16, N16 * sizeof(u64));
    if (!ok) return;
    const size_t x_at = ((size_t)b * beta * rows + t) * N16 + blk * 512, key_at = (size_t)pt * N16 + blk * 512 + 2 * lane;
    if (t >= level) {
        int_rows(S, s0, s1, o0, o1, pcs[pt], x_at + 2 * lane, (size_t)rows * N16, key_at, (size_t)np * N16, beta, accumulate);
        return;
    }
    u64* sm = sm_all + warp * ROW_SMEM;
    const u64* sp = sm + 2 * lane + 2 * (lane >> 3);    // the pair 2 lane (+ 64 j) of the padded buffer
    const FpRow r{twf + (size_t)t * N16, pcs[t].qd, pcs[t].qinvd};
    const double q = r.q, qinv = r.qinv;
    double f0[16], f1[16];
#pragma unroll
    for (int k = 0; k < 8; k++) {
        f0[2 * k] = f0[2 * k + 1] = f1[2 * k] = f1[2 * k + 1] = 0.0;
        if (accumulate) {
            const ulonglong2 v0 = *reinterpret_cast<const ulonglong2*>(o0 + 64 * k), v1 = *reinterpret_cast<const ulonglong2*>(o1 + 64 * k);
            f0[2 * k] = fp_load(v0.x, q), f0[2 * k + 1] = fp_load(v0.y, q);
            f1[2 * k] = fp_load(v1.x, q), f1[2 * k + 1] = fp_load(v1.y, q);
        }
    }
    uint32_t n = 0;
    for (uint32_t s = s0; s < s1; s++) {
        const u64* row = S.s[s].ext + x_at;
        const u64* key = S.s[s].key + key_at;
#pragma unroll 1
        for (uint32_t j = 0; j < beta; j++, row += (size_t)rows * N16, key += (size_t)2 * np * N16) {
            // the next digit's points and this digit's key words arrive in L2 while the digit is transformed (6.2 -> 5.8 ms below)
            if (j + 1 < beta) prefetch_l2(row + (size_t)rows * N16 + 16 * lane);
            prefetch_l2(key + 14 * lane);
            prefetch_l2(key + (size_t)np * N16 + 14 * lane);
            if (j != own) {
                const u64* in = row + 256 * (lane >> 4) + (lane & 15);
                double x[16];
#pragma unroll
                for (int k = 0; k < 16; k++) x[k] = FpRow::value(in[16 * k]);
                __syncwarp();                           // the previous digit's values have been read
                fwd_rows(r, x, sm, blk, lane);
            }
            // |x| <= q/2 once folded: products below 0.7 q, seven and a rest of q/2 below 8 q
            const bool fold = ++n % 7 == 0;
#pragma unroll
            for (int k = 0; k < 8; k++) {
                const ulonglong2 w0 = __ldg(reinterpret_cast<const ulonglong2*>(key + 64 * k));
                const ulonglong2 w1 = __ldg(reinterpret_cast<const ulonglong2*>(key + (size_t)np * N16 + 64 * k));
                double xa, xb;
                if (j != own) {
                    const ulonglong2 v = *reinterpret_cast<const ulonglong2*>(sp + 72 * k);
                    xa = r.fold(FpRow::value(v.x)), xb = r.fold(FpRow::value(v.y));
                } else {
                    const ulonglong2 v = *reinterpret_cast<const ulonglong2*>(row + 2 * lane + 64 * k);
                    xa = FpRow::value(v.x), xb = FpRow::value(v.y);
                }
                f0[2 * k] += fp_modmul(xa, fp_from_u64(w0.x), q, qinv);
                f0[2 * k + 1] += fp_modmul(xb, fp_from_u64(w0.y), q, qinv);
                f1[2 * k] += fp_modmul(xa, fp_from_u64(w1.x), q, qinv);
                f1[2 * k + 1] += fp_modmul(xb, fp_from_u64(w1.y), q, qinv);
            }
            if (fold) {
                fold16(r, f0);
                fold16(r, f1);
            }
        }
    }
#pragma unroll
    for (int k = 0; k < 8; k++) {
        *reinterpret_cast<ulonglong2*>(o0 + 64 * k) = make_ulonglong2(fp_store(f0[2 * k], q, qinv), fp_store(f0[2 * k + 1], q, qinv));
        *reinterpret_cast<ulonglong2*>(o1 + 64 * k) = make_ulonglong2(fp_store(f1[2 * k], q, qinv), fp_store(f1[2 * k + 1], q, qinv));
    }
}

int rows_inner_launch(fesc_ctx* ctx, const InnerSrcs& S, u64* acc, uint32_t level, uint32_t batch, int accumulate, bool separate, cudaStream_t st) {
    const uint32_t beta = (level + ctx->alpha - 1) / ctx->alpha;
    const dim3 grid((128 * batch + RI_WARPS - 1) / RI_WARPS, level + ctx->n_p, separate ? S.n : 1);
    launch(k_rows_inner, grid, 32 * RI_WARPS, 0, st, S, acc, ctx->d_twf, ctx->d_pc, level, ctx->n_q, ctx->n_p, ctx->alpha, beta, batch, accumulate,
           separate ? 1 : 0);
    FESC_CHECK_CUDA(ctx, cudaGetLastError());
    return FESC_OK;
}

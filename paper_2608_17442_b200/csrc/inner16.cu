// Key inner product fused with the last pass of the forward transform (N = 2^16, rows on primes below 2^50):
//   acc[b][p][t] = sum_s sum_j NTT(ext_s[b][j][t]) * key_s[j][p][t]
// for key switches whose converted digits serve one key only (rotations, relinearisation, giant-step sums; hoisted rotations keep
// the transformed digits for several keys).  The transformed rows are never stored: 75 MB written and 88 MB read per ciphertext at
// 24 limbs.
//
// What bounds it: the dispatch port (issue slots 50 %, FP64 pipe 47 %, its instructions hold the port for two or three cycles) at 16 warps
// per SM; 16 rotations at 24 limbs 0.77 -> 0.63 ms when the next digit's points and key words came to be fetched by bulk copies, while a
// digit is transformed: a warp's 4 KB of points and the CTA's 8 KB of keys (one copy for its ciphertexts) have their own shared memory and the
// L1 keeps the twiddles.  (Points by 8-byte asynchronous copies instead 1.2 ms, points alone by bulk copies 0.15 ms more.)
//
// The special rows arrive transformed and are multiplied by the last CTAs of the same launch: their products and loads run beside the
// data rows' arithmetic and fill its last wave (5.36 + 0.98 ms in two launches, 5.84 ms in one; first instead of last 6.02).  Two warps per 512 points with
// half the digits each, for single ciphertexts: 103 us against 86.  Where the division by P follows, the special rows are left after the first
// pass of their inverse transform, on the 512 points that a warp has just summed: 0.071 ms of a launch for 0.057 here.
//
// A warp owns 512 points of one row of one ciphertext.  It runs rounds C and D of every digit in turn (the digit that holds the row
// itself needs no transform), multiplies with the two key words of each point and keeps both sums in registers; 128 registers, 16
// warps per SM.  The warps of a CTA (up to four, shared out evenly: 5 run as 3 + 2) are ciphertexts on the same points.  Every wait is bounded
// (status word 5).
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

#define RI_X 512                    // words of a warp's staged points
#define RI_WARP_WORDS (RI_X + ROW_SMEM)
#define RI_KEY_WORDS 1024
// bytes of shared memory for a CTA of `warps`: keys, per warp the staged points and the exchange buffer, barriers
#define RI_SMEM(warps) (8 * (RI_KEY_WORDS + (warps) * RI_WARP_WORDS + (warps) + 2))
// first pass of the inverse transform of 512 canonical points at o, which this lane's earlier stores have put there (words 2 lane + 64 j of the block)
__device__ __forceinline__ void int_rows_inv(const IntRow& r, u64* o, u64* sm, uint32_t blk, uint32_t lane) {
    u64* s = sm + 2 * lane + 2 * (lane >> 3);
#pragma unroll
    for (int j = 0; j < 8; j++) {
        const ulonglong2 v = *reinterpret_cast<const ulonglong2*>(o + 2 * lane + 64 * j);
        *reinterpret_cast<ulonglong2*>(s + 72 * j) = v;
    }
    __syncwarp();
    u64 x[16];
    inv_rows(r, x, sm, blk, lane);
    u64* d = o + 256 * (lane >> 4) + (lane & 15);
#pragma unroll
    for (int k = 0; k < 16; k++) d[16 * k] = x[k];
    __syncwarp();
}

// itw: not nullptr where the sums are complete and the division by P takes the special rows after the first pass of their inverse transform
// (no launch for that pass, and its rows are still in L2)
__global__ void __launch_bounds__(32 * RI_WARPS, 4)
    k_rows_inner(InnerSrcs S, u64* acc, const double* __restrict__ twf, const ulonglong2* __restrict__ itw, const PrimeConst* __restrict__ pcs,
                 uint32_t level, uint32_t n_q, uint32_t K, uint32_t alpha, uint32_t beta, uint32_t batch, uint32_t groups, int accumulate, int sep,
                 uint32_t* __restrict__ status) {
    extern __shared__ __align__(128) u64 smem[];
    const uint32_t lane = threadIdx.x & 31, warp = threadIdx.x >> 5, warps = blockDim.x >> 5;
    const uint32_t blk = blockIdx.x / groups, b0 = (blockIdx.x - blk * groups) * warps, b = b0 + warp, t = blockIdx.y, rows = level + K, np = n_q + K;
    const uint32_t pt = t < level ? t : n_q + (t - level), own = t / alpha;
    const uint32_t base = (uint32_t)__cvta_generic_to_shared(smem), bars = base + 8 * (RI_KEY_WORDS + warps * RI_WARP_WORDS);
    const uint32_t x_bar = bars + 8 * warp, key_full = bars + 8 * warps, last = (batch - b0 < warps ? batch - b0 : warps) - 1;
    if (threadIdx.x == 0) {
        for (uint32_t i = 0; i <= warps; i++) mbar_init(bars + 8 * i, 1);
        smem[RI_KEY_WORDS + warps * RI_WARP_WORDS + warps + 1] = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    pdl_begin();
    __syncthreads();
    if (b >= batch) return;
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
        if (itw) {
            const IntRow r{itw + (size_t)pt * N16, pcs[pt].q, 2 * pcs[pt].q};
            u64* buf = smem + RI_KEY_WORDS + warp * RI_WARP_WORDS + RI_X;
#pragma unroll 1
            for (int p = 0; p < 2; p++) int_rows_inv(r, (p ? o1 : o0) - 2 * lane, buf, blk, lane);
        }
        return;
    }
    const uint32_t total = (s1 - s0) * beta;
    auto load_x = [&](uint32_t s, uint32_t j) {         // lane 0
        mbar_expect_tx(x_bar, 8 * RI_X);
        bulk_g2s(base + 8 * (RI_KEY_WORDS + warp * RI_WARP_WORDS), S.s[s].ext + x_at + (size_t)j * rows * N16, 8 * RI_X, x_bar);
    };
    auto load_keys = [&](uint32_t s, uint32_t j) {      // one lane of the CTA
        const u64* k = S.s[s].key + (size_t)pt * N16 + blk * 512 + (size_t)(2 * j) * np * N16;
        mbar_expect_tx(key_full, 8 * 1024);
        bulk_g2s(base, k, 8 * 512, key_full);
        bulk_g2s(base + 8 * 512, k + (size_t)np * N16, 8 * 512, key_full);
    };
    if (lane == 0) load_x(s0, 0);
    if (threadIdx.x == 0) load_keys(s0, 0);
    const u64* sx = smem + RI_KEY_WORDS + warp * RI_WARP_WORDS;
    u64* sm = smem + RI_KEY_WORDS + warp * RI_WARP_WORDS + RI_X;
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
    uint32_t s = s0, j = 0, room = accumulate || beta > 5 ? 4 : 5;
#pragma unroll 1
    for (uint32_t n = 0; n < total; n++) {
        const uint32_t s_next = j + 1 < beta ? s : s + 1, j_next = j + 1 < beta ? j + 1 : 0;
        if (mbar_wait_bounded(x_bar, n & 1)) {          // gives up: the other copy in flight is waited for as well (bounded)
            if (lane == 0) atomicExch(status, 5u);
            mbar_wait_bounded(key_full, n & 1);
            return;
        }
        if (j != own) {
            const u64* in = sx + 256 * (lane >> 4) + (lane & 15);
            double x[16];
#pragma unroll
            for (int k = 0; k < 16; k++) x[k] = FpRow::value(in[16 * k]);
            __syncwarp();                               // the staged points and the previous digit's values have been read
            if (lane == 0 && n + 1 < total) {
                before_refill();
                load_x(s_next, j_next);
            }
            fwd_rows<false>(r, x, sm, blk, lane);
        }
        if (mbar_wait_bounded(key_full, n & 1)) {
            if (lane == 0) atomicExch(status, 5u);
            if (j != own && n + 1 < total) mbar_wait_bounded(x_bar, (n + 1) & 1);
            return;
        }
        const u64* key = smem + 2 * lane;
#pragma unroll
        for (int k = 0; k < 8; k++) {
            const double2 w0 = *reinterpret_cast<const double2*>(key + 64 * k);
            const double2 w1 = *reinterpret_cast<const double2*>(key + 512 + 64 * k);
            const double2 v = *reinterpret_cast<const double2*>(j != own ? sp + 72 * k : sx + 2 * lane + 64 * k);
            f0[2 * k] += fp_modmul(v.x, w0.x, q, qinv);
            f0[2 * k + 1] += fp_modmul(v.y, w0.y, q, qinv);
            f1[2 * k] += fp_modmul(v.x, w1.x, q, qinv);
            f1[2 * k + 1] += fp_modmul(v.y, w1.y, q, qinv);
        }
        if (n + 1 < total) {
            __syncwarp();
            if (lane == 0) {
                before_refill();
                if (j == own) load_x(s_next, j_next);
                if (count_readers(key_full + 8, last) == last) load_keys(s_next, j_next);      // the last warp to have read the key words requests the next ones
            }
        }
        s = s_next, j = j_next;
        // A transformed point stays below 6.75 q, its product below 1.77 q, an own digit's below 0.6 q: four products and a rest of q/2 stay below
        // 8 q, and so do five that start from zero and have an own one among them (a source of up to five digits, or any first four)
        if (--room == 0 && n + 1 < total) {
            fold16(r, f0);
            fold16(r, f1);
            room = 4;
        }
    }
#pragma unroll
    for (int k = 0; k < 8; k++) {
        st_pair_once<true>(o0 + 64 * k, make_ulonglong2(fp_store(f0[2 * k], q, qinv), fp_store(f0[2 * k + 1], q, qinv)));
        st_pair_once<true>(o1 + 64 * k, make_ulonglong2(fp_store(f1[2 * k], q, qinv), fp_store(f1[2 * k + 1], q, qinv)));
    }
}

int rows_inner_launch(fesc_ctx* ctx, const InnerSrcs& S, u64* acc, uint32_t level, uint32_t batch, int accumulate, bool separate, bool inv_special,
                      cudaStream_t st) {
    const uint32_t beta = (level + ctx->alpha - 1) / ctx->alpha, groups = (batch + RI_WARPS - 1) / RI_WARPS, warps = (batch + groups - 1) / groups;
    const dim3 grid(128 * groups, level + ctx->n_p, separate ? S.n : 1);
    FESC_CHECK_CUDA(ctx, cudaFuncSetAttribute(k_rows_inner, cudaFuncAttributeMaxDynamicSharedMemorySize, RI_SMEM(RI_WARPS)));
    // Shared memory for four CTAs of four warps and no more: CTAs of one or two warps would fill all of it and leave the L1 too small for their twiddles
    // (one rotation of 24 limbs 254.6 -> 244.9 us, two 395 -> 379; three and more the same, with a smaller share 3 % slower).
    const int share = (int)((400 * (RI_SMEM(RI_WARPS) + 1024) + 228 * 1024 - 1) / (228 * 1024));
    FESC_CHECK_CUDA(ctx, cudaFuncSetAttribute(k_rows_inner, cudaFuncAttributePreferredSharedMemoryCarveout, share));
    launch(k_rows_inner, grid, 32 * warps, RI_SMEM(warps), st, S, acc, ctx->d_twf,
           inv_special ? ctx->d_itw : nullptr, ctx->d_pc, level, ctx->n_q, ctx->n_p, ctx->alpha, beta, batch, groups,
           accumulate, separate ? 1 : 0, ctx->d_status);
    FESC_CHECK_CUDA(ctx, cudaGetLastError());
    return FESC_OK;
}

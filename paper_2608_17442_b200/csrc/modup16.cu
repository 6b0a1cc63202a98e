// ModUp fused with the first pass of the forward transform (N = 2^16, data primes below 2^50, at most 4 limbs per digit).
//
// Per digit j and target modulus q_t:  ext_t = sum_a y_a m_a mod q_t,  y_a = d_a (Q_j/q_a)^-1 mod q_a (left by the inverse
// transform, whose last stage multiplies by N^-1 (Q_j/q_a)^-1),  m_a = (Q_j/q_a) mod q_t.  The converted rows are formed in
// the registers of the transform's first eight stages: they never exist in memory, which saves writing and reading
// (level + K - n_src) rows per digit.
//
// The sum is an exact mixed-pipe product: its quotient c = rint(sum_a y_a (m_a / q)) comes from the FP64 pipe (one
// multiply-add per term, m centred; its roundings add up to 2.51 at most, see convert4, so |v| <= 2.51 q < 2^63), its value
// v = sum_a y_a m_a - c q from wrapping 64-bit integer products on the multiplier pipe, which the FP64 butterflies leave idle.
//
// A CTA owns 4 columns of one digit of one ciphertext: the source columns (8 KB per limb) are read once into shared memory
// and serve all targets; six groups of 64 threads take targets from a counter, the slower rows on the 60-bit primes first.
//
// The first stage of the transform has one twiddle, so the constants of the lower half of the points carry it: those words are converted to
// their product, and the stage is additions only.
//
// What bounds it: the dispatch of wide operands (an FP64 multiply-add of three registers holds its port for three cycles), which
// conversion and butterflies share; 0.36 us per converted row at 24 limbs and 16 ciphertexts against 0.41 for a conversion kernel
// and a first pass of their own, and 1.2 GB less traffic per launch.  8 columns with 6 groups 0.38, division by P 0.39 against 0.33 ms; four exact
// FP64 products per word instead of the mixed sum 0.53 (the rounding unit takes nine cycles per product); byte planes on the tensor
// cores, eight targets at a time through shared memory, 0.45; the same for the division by P 0.51 against 0.36 unfused.
#define FESC_DBG_FILE 12   // file id in the sites a debug build reports
#include "ntt16.cuh"
#include "ops.cuh"

#define MU_GROUPS 6
#define MU_COLS 4
#define MU_TARGET_THREADS (MU_COLS * 16)
#define MU_THREADS (MU_GROUPS * MU_TARGET_THREADS)
#define MU_SRC (256 * MU_COLS)      // words of one source limb's columns

struct GroupBarrier {
    uint32_t id;
    __device__ __forceinline__ void operator()() const { asm volatile("bar.sync %0, %1;" ::"r"(id), "n"(MU_TARGET_THREADS) : "memory"); }
};

#define FP_MAGIC 6755399441055744.0      // 1.5 * 2^52: the low mantissa bits of FP_MAGIC + c hold the integer c, |c| < 2^51
#define FP_MAGIC_HI 0x43380000u

// v[0..3] = sum_a y_a m_a - c q (two's complement) for the points p, p + 16 MU_COLS, ... of the source columns.  The columns hold
// the doubles 2^52 + y, whose low 50 bits are y: one word serves both pipes without a conversion.  What 2^52 adds to the FP64 sum is
// in its starting value c0, what the exponent bits add to the cross products (weight 2^32, modulo 2^32) is taken off at the end.
// How far c is from the quotient, for any four primes below 2^50 (|m / q| <= 1/2, y < 2^50): the running sum starts at -2^52 sum(m / q)
// and loses 2^52 m / q with every term, so it is below 2^53, 2^53, 2^52 + 2^50, 2^52 and 2^51 in turn and the roundings (of the start and of
// four multiply-adds) are at most 1/2, 1/2, 1/2, 1/4 and 1/8; m / q as a double is off by 2^-55 at most, 1/32 per term after the product
// with y (what 2^52 makes of it is in c0, which is formed from the same doubles); the quotient rounds by 1/2.  Together 2.5.
template <int A>
__device__ __forceinline__ void convert4(const u64* p, uint32_t n_src, const ModUpTerm (*__restrict__ term)[FESC_MAX_PRIMES], uint32_t pt,
                                         double c0, u64 q, u64* v) {
    u64 acc[4];            // low product words, and the cross terms of weight 2^32 apart from them
    uint32_t cross[4], msum = 0;
    double s[4];
#pragma unroll
    for (int e = 0; e < 4; e++) acc[e] = 0, cross[e] = 0, s[e] = c0;
#pragma unroll
    for (int a = 0; a < A; a++) {
        if (a >= n_src) break;
        const ulonglong2 t = __ldg(reinterpret_cast<const ulonglong2*>(&term[a][pt]));
        const uint32_t ml = (uint32_t)t.x, mh = (uint32_t)(t.x >> 32);
        const double mq = __longlong_as_double((long long)t.y);
        msum += ml;
#pragma unroll
        for (int e = 0; e < 4; e++) {
            const u64 y = p[a * MU_SRC + e * 16 * MU_COLS];
            const uint32_t yl = (uint32_t)y, yh = (uint32_t)(y >> 32);
            s[e] = __fma_rn(__longlong_as_double((long long)y), mq, s[e]);
            asm("mad.wide.u32 %0, %1, %2, %0;" : "+l"(acc[e]) : "r"(yl), "r"(ml));
            asm("mad.lo.u32 %0, %1, %2, %0;" : "+r"(cross[e]) : "r"(yl), "r"(mh));
            asm("mad.lo.u32 %0, %1, %2, %0;" : "+r"(cross[e]) : "r"(yh), "r"(ml));
        }
    }
    const u64 nq = 0 - q;
    const uint32_t ql = (uint32_t)nq, qh = (uint32_t)(nq >> 32), corr = 0u - 0x43300000u * msum - FP_MAGIC_HI * ql;      // the exponent bits of y and c
#pragma unroll
    for (int e = 0; e < 4; e++) {
        const u64 c = (u64)__double_as_longlong(__dadd_rn(s[e], FP_MAGIC));
        const uint32_t cl = (uint32_t)c, ch = (uint32_t)(c >> 32);
        asm("mad.wide.u32 %0, %1, %2, %0;" : "+l"(acc[e]) : "r"(cl), "r"(ql));
        const uint32_t hi = (uint32_t)(acc[e] >> 32) + (cross[e] + corr + cl * qh + ch * ql);
        v[e] = ((u64)hi << 32) | (uint32_t)acc[e];
    }
}

template <int A>
__global__ void __launch_bounds__(MU_THREADS, 2)
    k_modup_cols(const u64* y, u64* ext, const ModUpDigit* __restrict__ tab, const double* __restrict__ twf,
                 const ulonglong2* __restrict__ tw, const PrimeConst* __restrict__ pcs, uint32_t level, uint32_t n_q, uint32_t K,
                 uint32_t beta) {
    pdl_begin();
    extern __shared__ __align__(16) u64 smem[];      // [A][MU_SRC] source columns, then one exchange buffer per group
    __shared__ uint32_t next, taken[2][MU_GROUPS];
    const uint32_t tid = threadIdx.x, tile = blockIdx.x, j = blockIdx.y, b = blockIdx.z;
    const ModUpDigit* dg = tab + j;
    const uint32_t first = dg->first, n_src = dg->n_src, rows = level + K, others = rows - n_src;
    const u64* src = y + ((size_t)b * level + first) * N16 + tile * MU_COLS;
    u64* out = ext + ((size_t)b * beta + j) * rows * N16 + tile * MU_COLS;
    if (!DBG_REGION(dg, sizeof(ModUpDigit)) || !DBG_REGION(src - tile * MU_COLS, (size_t)n_src * N16 * sizeof(u64)) ||
        !DBG_REGION(out - tile * MU_COLS, (size_t)rows * N16 * sizeof(u64)))
        return;                                     // the same for the whole CTA
    for (uint32_t i = tid; i < n_src * (MU_SRC / 2); i += MU_THREADS) {
        const uint32_t a = i / (MU_SRC / 2), r = (i / (MU_COLS / 2)) & 255, c = 2 * (i % (MU_COLS / 2));
        const ulonglong2 v = ld_pair_once<true>(src + (size_t)a * N16 + r * 256 + c);
        *reinterpret_cast<ulonglong2*>(smem + a * MU_SRC + r * MU_COLS + c) =
            make_ulonglong2(v.x | 0x4330000000000000ull, v.y | 0x4330000000000000ull);
    }
    if (tid == 0) next = 0;
    __syncthreads();
    const uint32_t group = tid / MU_TARGET_THREADS, gt = tid % MU_TARGET_THREADS, col = gt % MU_COLS, sub = gt / MU_COLS;
    const GroupBarrier bar{1 + group};
    u64* sm = smem + A * MU_SRC + group * COL_SMEM(MU_COLS);
    const u64* ys = smem + sub * MU_COLS + col;
    if (gt == 0) taken[0][group] = atomicAdd(&next, 1u);
    bar();
    // the next target is taken while this one is worked on; the exchange's barrier publishes it.  (A barrier before the exchange and not
    // at the head of the loop: a group's two warps may be half a target apart.)
    for (uint32_t slot = 0;; slot ^= 1) {
        const uint32_t o = taken[slot][group];
        if (o >= others) return;
        if (gt == 0) taken[slot ^ 1][group] = atomicAdd(&next, 1u);
        const uint32_t d = o < K ? 0 : o - K;
        const uint32_t t = o < K ? level + o : (d < first ? d : d + n_src), pt = o < K ? n_q + o : t;
        u64* p = out + (size_t)t * N16 + col;
        const u64 q = pcs[pt].q;
        if (q < FESC_FP_LIMIT) {
            FpRow r{twf + (size_t)pt * N16, pcs[pt].qd, pcs[pt].qinvd};
            double x[16];
#pragma unroll
            for (int k = 0; k < 16; k += 4) {
                u64 v[4];
                convert4<A>(ys + k * 16 * MU_COLS, n_src, dg->term[k / 8], pt, __ldg(&dg->start[k / 8][pt]), q, v);
#pragma unroll
                for (int e = 0; e < 4; e++) x[k + e] = __ll2double_rn((long long)v[e]);       // |v| <= 2.51 q, as COLS_MODUP takes them
            }
            fwd_cols<MU_COLS, COLS_MODUP>(r, x, sm, col, sub, bar);
#pragma unroll
            for (int k = 0; k < 16; k++) st_once(p + (16 * sub + k) * 256, FpRow::bits(x[k]));
        } else {
            const IntRow r{tw + (size_t)pt * N16, q, 2 * q};
            u64 x[16];
#pragma unroll
            for (int k = 0; k < 16; k += 4) {
                convert4<A>(ys + k * 16 * MU_COLS, n_src, dg->term[k / 8], pt, __ldg(&dg->start[k / 8][pt]), q, x + k);
#pragma unroll
                for (int e = 0; e < 4; e++) x[k + e] = csub(x[k + e] + 3 * q, r.q2);      // |v| <= 2.51 q: below 4q
            }
            fwd_cols<MU_COLS, COLS_MODUP>(r, x, sm, col, sub, bar);
#pragma unroll
            for (int k = 0; k < 16; k++) st_once(p + (16 * sub + k) * 256, x[k]);
        }
    }
}

bool modup16_supported(const fesc_ctx* ctx, uint32_t level) {
    if (ctx->log_n != 16 || ctx->alpha > 4 || ctx->n_p > 4) return false;
    for (uint32_t i = 0; i < level; i++)
        if (ctx->q[i] >= FESC_FP_LIMIT) return false;
    for (uint32_t k = 0; k < ctx->n_p; k++)
        if (ctx->q[ctx->n_q + k] >= (1ull << 61)) return false;
    return true;
}

template <int A>
static int launch_modup(fesc_ctx* ctx, const u64* y, u64* ext, uint32_t level, uint32_t batch, cudaStream_t st) {
    const uint32_t beta = (level + ctx->alpha - 1) / ctx->alpha, tiles = 256 / MU_COLS;
    const size_t smem = ((size_t)A * MU_SRC + MU_GROUPS * COL_SMEM(MU_COLS)) * sizeof(u64);
    auto kern = k_modup_cols<A>;
    FESC_CHECK_CUDA(ctx, cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    // One CTA takes all targets of a tile, however few tiles there are: shared by two to four CTAs, each of which loads the sources again, one rotation of
    // 24 / 15 / 9 / 5 limbs takes 267-275 / 187-195 / 150-162 / 109-111 us against 266 / 181 / 149 / 107, four of 15 limbs 444-469 against 419.
    launch(kern, dim3(tiles, beta, batch), MU_THREADS, smem, st, y, ext, ctx->tabs.d_modup + (size_t)(level - 1) * ctx->beta_max,
                                                                     ctx->d_twf, ctx->d_tw, ctx->d_pc, level, ctx->n_q, ctx->n_p, beta);
    return FESC_OK;
}
int modup16_cols_launch(fesc_ctx* ctx, const u64* y, u64* ext, uint32_t level, uint32_t batch, cudaStream_t st) {
    if (ctx->alpha <= 1) return launch_modup<1>(ctx, y, ext, level, batch, st);
    if (ctx->alpha <= 2) return launch_modup<2>(ctx, y, ext, level, batch, st);
    return launch_modup<4>(ctx, y, ext, level, batch, st);
}

// ---------------------------------------------------------------------------------------
// Division by P, conversion step fused with the first pass of the forward transform in the same way:
//   u_i = sum_k y_k m_k mod q_i,  y_k = r_k (P/p_k)^-1 mod p_k centred (the constant rides on the inverse transform's last stage),
//   m_k = (P/p_k) mod q_i.
// The sources have 60 bits, so the quotient is taken in units of 2^10: c = rint(sum_k y_k (m_k / (q 2^10))), |c| <= 2^50, and
// v = sum_k y_k m_k - c 2^10 q is below 5.2 2^10 q < 2^63; a second quotient from the high word of v leaves |v| <= 0.7 q.  A source word is
// kept once, with 2^59 added: its upper 52 bits below the exponent of 2^52 are the double that the quotient needs (a shift by eight in
// registers), the word itself goes to the integer products, what the additions contribute is in the sum's starting value and in the
// cross terms.  Reading the doubles as well loaded shared memory to 67 % and left room for three groups per CTA.
//
// How far c is from the quotient: the running sum stays within [0.75, 2.25] 2^52, so the start and the first three multiply-adds round by at most
// 1, the last by 1/2; the bits shifted out are below 1 each, times |m / 4q| <= 1/8; errors of m / 4q are below 2^-5.  Together 5.2.
// ---------------------------------------------------------------------------------------
#define MD_GROUPS 4
#define MD_THREADS (MD_GROUPS * MU_TARGET_THREADS)
#define MD_BIAS (1ull << 59)

// OPEN: the special rows await the last eight stages of their inverse transform, which are done here on the columns that the CTA
// needs anyway, one group per row: no pass of its own, 8 rows per ciphertext less to write and read (division of 42 rotations at 24 limbs,
// with the passes it replaces: 1.12 -> 0.98 ms).
template <int A, bool OPEN>
__global__ void __launch_bounds__(MD_THREADS, 2)
    k_moddown_cols(const u64* acc, u64* u, const ModDownTab* __restrict__ tab, const double* __restrict__ twf,
                   const ulonglong2* __restrict__ itw, const InvScale* __restrict__ scale, const PrimeConst* __restrict__ pcs, uint32_t level, uint32_t n_q, uint32_t K, uint32_t splits) {
    pdl_begin();
    extern __shared__ __align__(16) u64 smem[];      // [A][MU_SRC] sources, then one exchange buffer per group
    __shared__ uint32_t next, taken[2][MD_GROUPS];
    const uint32_t tid = threadIdx.x, tile = blockIdx.x / splits, part = blockIdx.x % splits, bp = blockIdx.y;
    const u64* src = acc + ((size_t)bp * (level + K) + level) * N16 + tile * MU_COLS;
    u64* out = u + (size_t)bp * level * N16 + tile * MU_COLS;
    if (!DBG_REGION(tab, sizeof(ModDownTab)) || !DBG_REGION(src - tile * MU_COLS, (size_t)K * N16 * sizeof(u64)) ||
        !DBG_REGION(out - tile * MU_COLS, (size_t)level * N16 * sizeof(u64)))
        return;                                     // the same for the whole CTA
    const uint32_t group = tid / MU_TARGET_THREADS, gt = tid % MU_TARGET_THREADS, col = gt % MU_COLS, sub = gt / MU_COLS;
    const GroupBarrier bar{1 + group};
    u64* sm = smem + A * MU_SRC + group * COL_SMEM(MU_COLS);
    if (OPEN) {
        for (uint32_t a = group; a < A; a += MD_GROUPS) {
            u64* y = smem + a * MU_SRC + sub * MU_COLS + col;
            if (a >= K) {
#pragma unroll
                for (int k = 0; k < 16; k++) y[k * 16 * MU_COLS] = MD_BIAS;
                continue;
            }
            const u64 p = pcs[n_q + a].q, half = tab->half[a];
            const IntRow r{itw + (size_t)(n_q + a) * N16, p, 2 * p};
            const InvScale& c = scale[n_q + a];
            u64 x[16];
#pragma unroll
            for (int k = 0; k < 16; k++) x[k] = ld_once(src + (size_t)a * N16 + (16 * sub + k) * 256 + col);
            bar();                                  // the buffer's last reader
            inv_cols<MU_COLS>(r, x, sm, col, sub, bar);
            const u64 n = c.n, ns = c.ns, nw = c.w, nws = c.ws;
#pragma unroll
            for (int k = 0; k < 8; k++) {           // as in ntt16_cols_inv
                const u64 e = x[k], v = x[k + 8], y0 = shoup(e + v, n, ns, p), y1 = shoup(e - v + r.q2, nw, nws, p);
                y[k * 16 * MU_COLS] = y0 + (y0 > half ? MD_BIAS - p : MD_BIAS);
                y[(k + 8) * 16 * MU_COLS] = y1 + (y1 > half ? MD_BIAS - p : MD_BIAS);
            }
        }
    } else {
        for (uint32_t i = tid; i < A * (MU_SRC / 2); i += MD_THREADS) {
            const uint32_t a = i / (MU_SRC / 2), r = (i / (MU_COLS / 2)) & 255, c = 2 * (i % (MU_COLS / 2)), at = a * MU_SRC + r * MU_COLS + c;
            ulonglong2 v = make_ulonglong2(MD_BIAS, MD_BIAS);
            if (a < K) {
                v = *reinterpret_cast<const ulonglong2*>(src + (size_t)a * N16 + r * 256 + c);
                const u64 p = pcs[n_q + a].q, half = tab->half[a];
                v.x += v.x > half ? MD_BIAS - p : MD_BIAS;
                v.y += v.y > half ? MD_BIAS - p : MD_BIAS;
            }
            *reinterpret_cast<ulonglong2*>(smem + at) = v;
        }
    }
    if (tid == 0) next = 0;
    __syncthreads();
    const u64* ys = smem + sub * MU_COLS + col;
    if (gt == 0) taken[0][group] = atomicAdd(&next, 1u);
    bar();
    for (uint32_t slot = 0;; slot ^= 1) {
        const uint32_t i = taken[slot][group] * splits + part;
        if (i >= level) return;
        if (gt == 0) taken[slot ^ 1][group] = atomicAdd(&next, 1u);
        const FpRow r{twf + (size_t)i * N16, pcs[i].qd, pcs[i].qinvd};
        const u64 nq = 0 - pcs[i].q, nq10 = nq << 10;
        const uint32_t ql = (uint32_t)nq, qh = (uint32_t)(nq >> 32), tl = (uint32_t)nq10, th = (uint32_t)(nq10 >> 32);
        const uint32_t corr2 = 0u - FP_MAGIC_HI * ql;
        const double q32 = 4294967296.0 * r.qinv;
        double x[16];
#pragma unroll
        for (int k = 0; k < 16; k += 4) {
            u64 v[4];
            uint32_t cross[4], msum = 0;
            double s[4];
#pragma unroll
            for (int e = 0; e < 4; e++) v[e] = 0, cross[e] = 0, s[e] = __ldg(&tab->start[k / 8][i]);
#pragma unroll
            for (int a = 0; a < A; a++) {
                const ulonglong2 t = __ldg(reinterpret_cast<const ulonglong2*>(&tab->term[k / 8][a][i]));
                const uint32_t ml = (uint32_t)t.x, mh = (uint32_t)(t.x >> 32);
                const double mq = __longlong_as_double((long long)t.y);
                msum += ml;
#pragma unroll
                for (int e = 0; e < 4; e++) {
                    const u64 y = ys[a * MU_SRC + (k + e) * 16 * MU_COLS];
                    const uint32_t yl = (uint32_t)y, yh = (uint32_t)(y >> 32);
                    s[e] = __fma_rn(__hiloint2double((int)(0x43300000u + (yh >> 8)), (int)__funnelshift_r(yl, yh, 8)), mq, s[e]);
                    asm("mad.wide.u32 %0, %1, %2, %0;" : "+l"(v[e]) : "r"(yl), "r"(ml));
                    asm("mad.lo.u32 %0, %1, %2, %0;" : "+r"(cross[e]) : "r"(yl), "r"(mh));
                    asm("mad.lo.u32 %0, %1, %2, %0;" : "+r"(cross[e]) : "r"(yh), "r"(ml));
                }
            }
#pragma unroll
            for (int e = 0; e < 4; e++) {
                const uint32_t corr = 0u - (msum << 27) - FP_MAGIC_HI * tl;      // the bias times the sum of m; the exponent bits of c
                const u64 c = (u64)__double_as_longlong(s[e]);
                const uint32_t cl = (uint32_t)c, ch = (uint32_t)(c >> 32);
                asm("mad.wide.u32 %0, %1, %2, %0;" : "+l"(v[e]) : "r"(cl), "r"(tl));
                uint32_t hi = (uint32_t)(v[e] >> 32) + (cross[e] + cl * th + ch * tl + corr);
                // second quotient: the signed high word times 2^32 / q
                const double d = __int2double_rn((int)hi);
                const u64 c2 = (u64)__double_as_longlong(__fma_rn(d, q32, FP_MAGIC));
                const uint32_t dl = (uint32_t)c2, dh = (uint32_t)(c2 >> 32);
                u64 w = ((u64)hi << 32) | (uint32_t)v[e];
                asm("mad.wide.u32 %0, %1, %2, %0;" : "+l"(w) : "r"(dl), "r"(ql));
                hi = (uint32_t)(w >> 32) + (dl * qh + dh * ql + corr2);
                x[k + e] = __ll2double_rn((long long)((u64)hi << 32 | (uint32_t)w));
            }
        }
        fwd_cols<MU_COLS, COLS_MODDOWN>(r, x, sm, col, sub, bar);
        u64* p = out + (size_t)i * N16 + col;
#pragma unroll
        for (int k = 0; k < 16; k++) st_once(p + (16 * sub + k) * 256, FpRow::bits(x[k]));
    }
}

// special primes below 2^60 (|y| < 2^59), data primes of 2^40 to 2^50 (the second quotient ignores the low word of v)
bool moddown16_supported(const fesc_ctx* ctx, uint32_t level) {
    if (ctx->log_n != 16 || ctx->n_p > 4) return false;
    for (uint32_t i = 0; i < level; i++)
        if (ctx->q[i] >= FESC_FP_LIMIT || ctx->q[i] < (1ull << 40)) return false;
    for (uint32_t k = 0; k < ctx->n_p; k++)
        if (ctx->q[ctx->n_q + k] >= (1ull << 60)) return false;
    return true;
}
bool moddown16_open(const fesc_ctx* ctx, uint32_t level) {
    bool open = moddown16_supported(ctx, level);
    for (uint32_t k = 0; k < ctx->n_p; k++) open = open && ctx->q[ctx->n_q + k] >= FESC_FP_LIMIT;
    return open;
}
template <int A, bool OPEN>
static int launch_moddown(fesc_ctx* ctx, const u64* acc, u64* u, uint32_t level, uint32_t polys, cudaStream_t st) {
    const uint32_t tiles = 256 / MU_COLS;
    const size_t smem = ((size_t)A * MU_SRC + MD_GROUPS * COL_SMEM(MU_COLS)) * sizeof(u64);
    auto kern = k_moddown_cols<A, OPEN>;
    FESC_CHECK_CUDA(ctx, cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    // Two CTAs share the limbs of a tile for the two polynomials of one ciphertext, which would leave more than half of the places (two per SM) empty
    // otherwise.  Each opens the special rows again, which costs as much as a third of 24 limbs: one rotation of 24 / 15 / 9 / 5 limbs with 1, 2, 4 CTAs per tile 277, 260, 271 / 194, 188, 194 / 155, 147, 160 /
    // 114, 106, 113 us; two: 395, 400, 416 / 250, 257, 269 / 195, 205, 219 / 138, 150, 163; eight of 24 limbs 1239, 1265, 1341.
    const uint32_t splits = polys <= 2 ? 2 : 1;
    launch(kern, dim3(tiles * splits, polys), MD_THREADS, smem, st, acc, u, ctx->tabs.d_moddown, ctx->d_twf, ctx->d_itw, ctx->tabs.d_down_scale, ctx->d_pc,
           level, ctx->n_q, ctx->n_p, splits);
    return FESC_OK;
}
template <int A>
static int launch_moddown(fesc_ctx* ctx, const u64* acc, u64* u, uint32_t level, uint32_t polys, cudaStream_t st) {
    return moddown16_open(ctx, level) ? launch_moddown<A, true>(ctx, acc, u, level, polys, st) : launch_moddown<A, false>(ctx, acc, u, level, polys, st);
}
int moddown16_cols_launch(fesc_ctx* ctx, const u64* acc, u64* u, uint32_t level, uint32_t polys, cudaStream_t st) {
    if (ctx->n_p <= 1) return launch_moddown<1>(ctx, acc, u, level, polys, st);
    if (ctx->n_p <= 2) return launch_moddown<2>(ctx, acc, u, level, polys, st);
    return launch_moddown<4>(ctx, acc, u, level, polys, st);
}

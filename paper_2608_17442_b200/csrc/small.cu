// Rings N = 2^10 .. 2^12: transforms and whole key-switch steps of one row per CTA.
//
// A row (8 to 32 KB) fits one CTA: N/8 threads keep eight points each and run the transform as register rounds of 3, 3, 3 and
// log N - 9 stages with three exchanges through shared memory.  At these sizes a call is a few hundred thousand products and
// its time is launches and latencies, so every step around a transform is done by the CTA that holds the row.  Eight points a
// thread and not sixteen: a row is one CTA's chain of dependent instructions, and twice the warps hide twice as much of it (a product
// with a plaintext and two rotations of 4 / 40 / 200 ciphertexts of 3 limbs at N = 2^12: 95.2 -> 72.0, 137 -> 128, 697 -> 587 us).
//   k_small_coef    [permutation of c1, copy of its own rows] + inverse transform (times a constant)
//   k_small_modup   conversion of a digit to one target + forward transform
//   k_small_inner   key inner product of one row [+ inverse transform of the rows on special primes]
//   k_small_down    conversion of the special rows to one limb + forward transform + last step of the division [+ permuted c0]
//   k_small_rescale conversion of the last limb + forward transform + last step of the division
// A rotation takes 4 launches instead of 9, a rescale 2 instead of 5.
//   k_small_switch  the first four as one launch of clusters, for calls that leave most of the device idle (rule: switch_ctas)
#define FESC_DBG_FILE 2   // file id in the sites a debug build reports
#include "ntt16.cuh"
#include "ops.cuh"

// Point e of a row lies at SM_AT(e) of the buffer: its place among sixteen words is exchanged by bits 4..6 of e and their parity, so that the accesses
// of every round (stride N/8, N/64, N/512 and 1) reach sixteen different banks per half-warp.  (A word of padding per eight points left the
// accesses at consecutive words in two steps each: 300 polynomials of 3 limbs at N = 2^12, forward 25.0 us with it and 22.8 so, inverse 29.6 and 27.8.)
// The map is linear over exclusive or, and the thread's and the register's parts of e share no bit.
#define SM_AT(e) ((e) ^ (((e) >> 4) & 7) ^ (((((e) >> 4) ^ ((e) >> 5) ^ ((e) >> 6)) & 1) << 3))
// dynamic shared memory: the row, then a copy of the row's twiddle table (8 bytes per entry for FP64 rows, 16 for integer
// rows).  The copy is made before the kernel waits for its predecessor: at these sizes a stage's twiddles fetched from L2 one
// stage at a time cost more than its butterflies.
#define SM_ROW(LOG) (1u << LOG)
#define SM_BYTES(LOG) (8 * (SM_ROW(LOG) + 2 * (1u << LOG)))
// CTAs per SM that their shared memory leaves room for.  A rescale takes its 64 registers for it: 150 ciphertexts of 3 limbs at N = 2^12 41.4 us with 74
// registers and one CTA per SM, 33.8 so.
#define SM_CTAS(LOG) (32 >> ((LOG) - 8))
typedef FpRowT<true> FpS;
typedef IntRowT<true> IntS;
template <int LOG>
__device__ __forceinline__ void small_tables(u64* sm, const SmallTables& tb, uint32_t pi, bool inv) {
    constexpr uint32_t N = 1u << LOG, T = N / 8;
    ulonglong2* dst = reinterpret_cast<ulonglong2*>(sm + SM_ROW(LOG));
    if (tb.pc[pi].q < FESC_FP_LIMIT) {
        const ulonglong2* src = reinterpret_cast<const ulonglong2*>((inv ? tb.itwf : tb.twf) + (size_t)pi * N);
#pragma unroll
        for (int k = 0; k < 4; k++) dst[k * T + threadIdx.x] = __ldg(src + k * T + threadIdx.x);
    } else {
        const ulonglong2* src = (inv ? tb.itw : tb.tw) + (size_t)pi * N;
#pragma unroll
        for (int k = 0; k < 8; k++) dst[k * T + threadIdx.x] = __ldg(src + k * T + threadIdx.x);
    }
}
// (No __restrict__ on buffers that kernels write: see pdl_begin.)
// The next kernel is let in after the wait and not before it: a kernel that still waits would let in the one after it, whose CTAs then sit on the SMs
// that the first one's are to run on.  Rescales one after the other of 16 ciphertexts of 3 limbs at N = 2^12 17.8 us with the trigger first, 10.8 so; of
// 40 of 6 limbs at N = 2^11 12.3 and 10.9; a rotation of one ciphertext of 2 limbs at N = 2^10 in four launches 30.8 and 25.1.
#define SMALL_BEGIN(used, pi, inv)                                  \
    extern __shared__ __align__(16) u64 sm[];                       \
    if (used) small_tables<LOG>(sm, tb, pi, inv);                   \
    asm volatile("griddepcontrol.wait;" ::: "memory");              \
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");

// Stage S (0..2) of a round on eight registers: distance 4 >> S, twiddles (i0 << S) + j for the j-th group.  FOLD: as in fwd_stage.
template <int S, bool FOLD, class R>
__device__ __forceinline__ void fwd8(const R& r, typename R::T (&x)[8], uint32_t i0) {
    typename R::W w[8];
    r.template load<S>(w, i0 << S);
    constexpr int d = 4 >> S;
#pragma unroll
    for (int k = 0; k < 4; k++) {
        const int i = (k / d) * 2 * d + k % d;
        if (FOLD) x[i] = r.fold(x[i]);
        r.ct(x[i], x[i + d], w[k / d]);
    }
}
template <int S, class R>
__device__ __forceinline__ void inv8(const R& r, typename R::T (&x)[8], uint32_t i0) {
    typename R::W w[8];
    r.template load<S>(w, i0 << S);
    constexpr int d = 4 >> S;
#pragma unroll
    for (int k = 0; k < 4; k++) {
        const int i = (k / d) * 2 * d + k % d;
        r.gs(x[i], x[i + d], w[k / d]);
    }
}
template <class R>
__device__ __forceinline__ void fold8(const R& r, typename R::T (&x)[8]) {
#pragma unroll
    for (int k = 0; k < 8; k++) x[k] = r.fold(x[k]);
}
// position in the buffer of point k of a thread in the rounds of stride N/8 (1), N/64 (2), N/512 (3) and 1 (4)
template <int LOG, int ROUND>
__device__ __forceinline__ uint32_t at8(uint32_t k) {
    constexpr uint32_t N = 1u << LOG, L = ROUND == 1 ? N / 8 : ROUND == 2 ? N / 64 : ROUND == 3 ? N / 512 : 1;
    const uint32_t t = threadIdx.x / L * 8 * L + threadIdx.x % L;
    return ROUND == 1 ? k * L + SM_AT(t) : (SM_AT(t) ^ (SM_AT(k * L) & 15)) + (SM_AT(k * L) & ~15u);
}
// Forward: x[k] = point k N/8 + tid on entry, up to q; on return the buffer holds the transformed row, unreduced.  Six stages reach
// 7.62 q; the folded seventh leaves 2.43, the eleventh 7.47, the folded twelfth 2.40 q.
template <int LOG, class R>
__device__ __forceinline__ void small_fwd(const R& r, typename R::T (&x)[8], u64* sm) {
    constexpr uint32_t N = 1u << LOG, L2 = N / 64, L3 = N / 512;
    constexpr int S = LOG - 9;
    const uint32_t tid = threadIdx.x;
    __syncthreads();               // the twiddle table is complete
    fwd8<0, false>(r, x, 1);
    fwd8<1, false>(r, x, 1);
    fwd8<2, false>(r, x, 1);
#pragma unroll
    for (int k = 0; k < 8; k++) sm[at8<LOG, 1>(k)] = R::bits(x[k]);
    __syncthreads();
#pragma unroll
    for (int k = 0; k < 8; k++) x[k] = R::value(sm[at8<LOG, 2>(k)]);
    fwd8<0, false>(r, x, 8 + tid / L2);
    fwd8<1, false>(r, x, 8 + tid / L2);
    fwd8<2, false>(r, x, 8 + tid / L2);
    // a thread writes the points it has read: no barrier needed before
#pragma unroll
    for (int k = 0; k < 8; k++) sm[at8<LOG, 2>(k)] = R::bits(x[k]);
    __syncthreads();
#pragma unroll
    for (int k = 0; k < 8; k++) x[k] = R::value(sm[at8<LOG, 3>(k)]);
    fwd8<0, true>(r, x, 64 + tid / L3);
    fwd8<1, false>(r, x, 64 + tid / L3);
    fwd8<2, false>(r, x, 64 + tid / L3);
#pragma unroll
    for (int k = 0; k < 8; k++) sm[at8<LOG, 3>(k)] = R::bits(x[k]);
    __syncthreads();
#pragma unroll
    for (int k = 0; k < 8; k++) x[k] = R::value(sm[at8<LOG, 4>(k)]);
#pragma unroll
    for (int s = 0; s < S; s++) {
        const int d = 1 << (S - 1 - s);
#pragma unroll
        for (int b = 0; b < 4 / d; b++) {
            typename R::W w;
            r.one(w, (512u << s) + ((8 * tid + 2 * d * b) >> (S - s)));
#pragma unroll
            for (int k = 0; k < d; k++) {
                if (s == 2) x[2 * d * b + k] = r.fold(x[2 * d * b + k]);
                r.ct(x[2 * d * b + k], x[2 * d * b + k + d], w);
            }
        }
    }
#pragma unroll
    for (int k = 0; k < 8; k++) sm[at8<LOG, 4>(k)] = R::bits(x[k]);
    __syncthreads();
}
// Three stages of an inverse round on words up to 2 q, and the same for two of the three (LAST: the third is the caller's).  A stage doubles
// the sums and leaves its products at (1/2 + 0.1875 B) q: after two stages words 0 and 4 may have reached 8 q and are folded; after three, words 1
// (5 q) and 2 (4 q) are, and the rest stay below 2 q.  (All eight words folded after every round:
// inverse transforms of 80 polynomials of 8 limbs at N = 2^11 10.3 us, so 9.9.)
template <bool LAST, class R>
__device__ __forceinline__ void inv_round(const R& r, typename R::T (&x)[8], uint32_t i0) {
    inv8<2>(r, x, i0);
    inv8<1>(r, x, i0);
    x[0] = r.fold(x[0]), x[4] = r.fold(x[4]);
    if (LAST) return;
    inv8<0>(r, x, i0);
    x[1] = r.fold(x[1]), x[2] = r.fold(x[2]);
}
// Inverse: the buffer holds the row on entry, centred (and a barrier has passed); x[k] = point k N/8 + tid on return, the last
// stage still to be done (pairs k, k + 4).
template <int LOG, class R>
__device__ __forceinline__ void small_inv(const R& r, typename R::T (&x)[8], u64* sm) {
    constexpr uint32_t N = 1u << LOG, L2 = N / 64, L3 = N / 512;
    constexpr int S = LOG - 9;
    const uint32_t tid = threadIdx.x;
#pragma unroll
    for (int k = 0; k < 8; k++) x[k] = R::value(sm[at8<LOG, 4>(k)]);
#pragma unroll
    for (int s = S - 1; s >= 0; s--) {
        const int d = 1 << (S - 1 - s);
#pragma unroll
        for (int b = 0; b < 4 / d; b++) {
            typename R::W w;
            r.one(w, (512u << s) + ((8 * tid + 2 * d * b) >> (S - s)));
#pragma unroll
            for (int k = 0; k < d; k++) r.gs(x[2 * d * b + k], x[2 * d * b + k + d], w);
        }
    }
    if (S == 3) x[0] = r.fold(x[0]), x[1] = r.fold(x[1]);      // 4 q and 2.75 q
#pragma unroll
    for (int k = 0; k < 8; k++) sm[at8<LOG, 4>(k)] = R::bits(x[k]);
    __syncthreads();
#pragma unroll
    for (int k = 0; k < 8; k++) x[k] = R::value(sm[at8<LOG, 3>(k)]);
    inv_round<false>(r, x, 64 + tid / L3);
#pragma unroll
    for (int k = 0; k < 8; k++) sm[at8<LOG, 3>(k)] = R::bits(x[k]);
    __syncthreads();
#pragma unroll
    for (int k = 0; k < 8; k++) x[k] = R::value(sm[at8<LOG, 2>(k)]);
    inv_round<false>(r, x, 8 + tid / L2);
#pragma unroll
    for (int k = 0; k < 8; k++) sm[at8<LOG, 2>(k)] = R::bits(x[k]);
    __syncthreads();
#pragma unroll
    for (int k = 0; k < 8; k++) x[k] = R::value(sm[at8<LOG, 1>(k)]);
    inv_round<true>(r, x, 1);
}
// last inverse stage of an FP64 / integer row with the constants `s` (nullptr: the plain ones), canonical words to o
template <int LOG>
__device__ __forceinline__ void small_inv_store(const FpS& r, double (&x)[8], const PrimeConst& pc, const InvScale* s, u64* o) {
    constexpr uint32_t T = (1u << LOG) / 8;
    const double n = s ? s->nd : pc.ninvd, w = s ? s->wd : pc.ninvwd;
#pragma unroll
    for (int k = 0; k < 4; k++) {
        const double u = x[k], v = x[k + 4];
        o[k * T + threadIdx.x] = fp_store(fp_modmul(u + v, n, r.q, r.qinv), r.q, r.qinv);
        o[(k + 4) * T + threadIdx.x] = fp_store(fp_modmul(u - v, w, r.q, r.qinv), r.q, r.qinv);
    }
}
template <int LOG>
__device__ __forceinline__ void small_inv_store(const IntS& r, u64 (&x)[8], const PrimeConst& pc, const InvScale* s, u64* o) {
    constexpr uint32_t T = (1u << LOG) / 8;
    const u64 n = s ? s->n : pc.ninv, ns = s ? s->ns : pc.ninvs, w = s ? s->w : pc.ninvw, ws = s ? s->ws : pc.ninvws;
#pragma unroll
    for (int k = 0; k < 4; k++) {
        const u64 u = x[k], v = x[k + 4];
        o[k * T + threadIdx.x] = shoup(u + v, n, ns, r.q);
        o[(k + 4) * T + threadIdx.x] = shoup(u - v + r.q2, w, ws, r.q);
    }
}
// inverse transform of the canonical row in the buffer (barrier passed) to o
template <int LOG>
__device__ __forceinline__ void small_inv_row(u64* sm, const SmallTables& tb, uint32_t pi, const InvScale* s, u64* o) {
    const PrimeConst& pc = tb.pc[pi];
    if (pc.q < FESC_FP_LIMIT) {
        const FpS r{reinterpret_cast<const double*>(sm + SM_ROW(LOG)), pc.qd, pc.qinvd};
#pragma unroll
        for (int k = 0; k < 8; k++) sm[at8<LOG, 4>(k)] = FpS::bits(fp_load(sm[at8<LOG, 4>(k)], r.q));
        double x[8];
        small_inv<LOG>(r, x, sm);
        small_inv_store<LOG>(r, x, pc, s, o);
    } else {
        const IntS r{reinterpret_cast<const ulonglong2*>(sm + SM_ROW(LOG)), pc.q, 2 * pc.q};
        u64 x[8];
        small_inv<LOG>(r, x, sm);
        small_inv_store<LOG>(r, x, pc, s, o);
    }
}

// ---------------------------------------------------------------------------------------
// plain transforms, one row per CTA (skipped rows launch nothing: RowList)
// ---------------------------------------------------------------------------------------
template <int LOG, bool INV>
__global__ void __launch_bounds__(1 << (LOG - 3)) k_small_ntt(u64* data, SmallTables tb, RowList list) {
    constexpr uint32_t N = 1u << LOG, T = N / 8;
    const uint32_t rep = blockIdx.x / list.count, e = blockIdx.x - rep * list.count, pi = list.prime[e], tid = threadIdx.x;
    SMALL_BEGIN(true, pi, INV)
    u64* p = data + ((size_t)rep * list.period + list.row[e]) * N;
    if (!DBG_REGION(p, N * sizeof(u64))) return;
    if (INV) {
#pragma unroll
        for (int k = 0; k < 8; k++) sm[at8<LOG, 1>(k)] = p[k * T + tid];
        __syncthreads();
        small_inv_row<LOG>(sm, tb, pi, nullptr, p);
        return;
    }
    const PrimeConst& pc = tb.pc[pi];
    if (pc.q < FESC_FP_LIMIT) {
        const FpS r{reinterpret_cast<const double*>(sm + SM_ROW(LOG)), pc.qd, pc.qinvd};
        double x[8];
#pragma unroll
        for (int k = 0; k < 8; k++) x[k] = fp_from_u64(p[k * T + tid]);
        small_fwd<LOG>(r, x, sm);
#pragma unroll
        for (int k = 0; k < 8; k++) p[k * T + tid] = fp_store(FpS::value(sm[at8<LOG, 1>(k)]), r.q, r.qinv);
    } else {
        const IntS r{reinterpret_cast<const ulonglong2*>(sm + SM_ROW(LOG)), pc.q, 2 * pc.q};
        u64 x[8];
#pragma unroll
        for (int k = 0; k < 8; k++) x[k] = p[k * T + tid];
        small_fwd<LOG>(r, x, sm);
#pragma unroll
        for (int k = 0; k < 8; k++) p[k * T + tid] = csub(csub(sm[at8<LOG, 1>(k)], r.q2), r.q);
    }
}

// ---------------------------------------------------------------------------------------
// grid (level, batch): the polynomial to be switched, src[b] = [level][N] EVAL, read through the permutation of g (0: none), its own
// rows kept in `own` (may be nullptr), COEFF rows times (Q_j/q)^-1 to dcoef.  src may be dcoef when g = 0.
// ---------------------------------------------------------------------------------------
template <int LOG>
__device__ __forceinline__ void coef_row(u64* sm, uint32_t l, uint32_t b, const u64* src, size_t src_stride, u64* own, size_t own_stride,
                                         uint32_t own_rows, uint32_t alpha, u64* dcoef, const SmallTables& tb, const InvScale* __restrict__ scale,
                                         uint32_t level, u64 g) {
    constexpr uint32_t N = 1u << LOG, T = N / 8;
    const uint32_t tid = threadIdx.x;
    const u64* in = src + (size_t)b * src_stride + (size_t)l * N;
    u64* o = dcoef + ((size_t)b * level + l) * N;
    u64* w = own ? own + (size_t)b * own_stride + ((size_t)(l / alpha) * own_rows + l) * N : nullptr;
    if (!DBG_REGION(in, N * sizeof(u64)) || !DBG_REGION(o, N * sizeof(u64)) || (w && !DBG_REGION(w, N * sizeof(u64)))) return;
#pragma unroll
    for (int k = 0; k < 8; k++) {
        const uint32_t t = k * T + tid;
        const u64 v = in[g ? galois_src(t, LOG, g) : t];
        sm[at8<LOG, 1>(k)] = v;
        if (w) w[t] = v;
    }
    __syncthreads();
    small_inv_row<LOG>(sm, tb, l, scale + l, o);
}
template <int LOG>
__global__ void __launch_bounds__(1 << (LOG - 3)) k_small_coef(const u64* src, size_t src_stride, u64* own, size_t own_stride, uint32_t own_rows,
                                                               uint32_t alpha, u64* dcoef, SmallTables tb, const InvScale* __restrict__ scale,
                                                               uint32_t level, u64 g) {
    SMALL_BEGIN(true, blockIdx.x, true)
    coef_row<LOG>(sm, blockIdx.x, blockIdx.y, src, src_stride, own, own_stride, own_rows, alpha, dcoef, tb, scale, level, g);
}

// grid (rows of all digits but the own ones, batch): ext[b][j][t] = NTT(sum_a y_a m_a)
template <int LOG>
__device__ __forceinline__ void modup_row(u64* sm, uint32_t j, uint32_t t, uint32_t pt, uint32_t b, const u64* y, u64* ext,
                                          const ModUpDigit* __restrict__ tab, const SmallTables& tb, uint32_t level, uint32_t rows, uint32_t beta) {
    constexpr uint32_t N = 1u << LOG, T = N / 8;
    const uint32_t tid = threadIdx.x;
    const ModUpDigit* dg = tab + j;
    const uint32_t n_src = dg->n_src;
    const u64* src = y + ((size_t)b * level + dg->first) * N + tid;
    u64* o = ext + (((size_t)b * beta + j) * rows + t) * N + tid;
    if (!DBG_REGION(src - tid, (size_t)n_src * N * sizeof(u64)) || !DBG_REGION(o - tid, N * sizeof(u64))) return;
    const PrimeConst& pc = tb.pc[pt];
    bool fp = pc.q < FESC_FP_LIMIT;
    for (uint32_t a = 0; a < n_src; a++) fp = fp && tb.pc[dg->first + a].q < FESC_FP_LIMIT;
    if (fp) {
        const FpS r{reinterpret_cast<const double*>(sm + SM_ROW(LOG)), pc.qd, pc.qinvd};
        double x[8];
#pragma unroll
        for (int k = 0; k < 8; k++) x[k] = 0.0;
        for (uint32_t a = 0; a < n_src; a++) {         // every product below 0.875 q, folded back after every third
            const double m = dg->matd[a][pt];
#pragma unroll
            for (int k = 0; k < 8; k++) x[k] += fp_modmul(fp_from_u64(src[(size_t)a * N + k * T]), m, r.q, r.qinv);
            if (a % 3 == 2) fold8(r, x);
        }
        if (n_src > 1) fold8(r, x);
        small_fwd<LOG>(r, x, sm);
#pragma unroll
        for (int k = 0; k < 8; k++) o[k * T] = fp_store(FpS::value(sm[at8<LOG, 1>(k)]), r.q, r.qinv);
        return;
    }
    u64 v[8];
#pragma unroll
    for (int k = 0; k < 8; k++) {
        acc128 s{0, 0};
        for (uint32_t a = 0; a < n_src; a++) mac128(s, src[(size_t)a * N + k * T], dg->mat[a][pt]);
        v[k] = reduce128(s.hi, s.lo, pc);
    }
    if (pc.q < FESC_FP_LIMIT) {
        const FpS r{reinterpret_cast<const double*>(sm + SM_ROW(LOG)), pc.qd, pc.qinvd};
        double x[8];
#pragma unroll
        for (int k = 0; k < 8; k++) x[k] = fp_from_u64(v[k]);
        small_fwd<LOG>(r, x, sm);
#pragma unroll
        for (int k = 0; k < 8; k++) o[k * T] = fp_store(FpS::value(sm[at8<LOG, 1>(k)]), r.q, r.qinv);
    } else {
        const IntS r{reinterpret_cast<const ulonglong2*>(sm + SM_ROW(LOG)), pc.q, 2 * pc.q};
        small_fwd<LOG>(r, v, sm);
#pragma unroll
        for (int k = 0; k < 8; k++) o[k * T] = csub(csub(sm[at8<LOG, 1>(k)], r.q2), r.q);
    }
}

template <int LOG>
__global__ void __launch_bounds__(1 << (LOG - 3)) k_small_modup(const u64* y, u64* ext, const ModUpDigit* __restrict__ tab,
                                                                SmallTables tb, uint32_t level, uint32_t n_q, uint32_t K, uint32_t alpha, uint32_t beta) {
    const uint32_t rows = level + K, j = blockIdx.x / rows, t = blockIdx.x - j * rows;
    if (t < level && t / alpha == j) return;
    const uint32_t pt = t < level ? t : n_q + (t - level);
    SMALL_BEGIN(true, pt, false)
    modup_row<LOG>(sm, j, t, pt, blockIdx.y, y, ext, tab, tb, level, rows, beta);
}

// grid (level + K, 2, batch): acc[b][p][t] = sum over sources and digits of ext . key (+ what acc holds); with `last` the rows on
// special primes are left as COEFF residues times (P/p_k)^-1
template <int LOG>
__device__ __forceinline__ void inner_row(u64* sm, uint32_t t, uint32_t pol, uint32_t pt, uint32_t b, const InnerSrcs& S, u64* acc, const SmallTables& tb,
                                          const InvScale* __restrict__ scale, uint32_t level, uint32_t n_q, uint32_t K, uint32_t beta, int accumulate,
                                          int last) {
    constexpr uint32_t N = 1u << LOG, T = N / 8;
    const uint32_t tid = threadIdx.x, rows = level + K;
    u64* o = acc + (((size_t)b * 2 + pol) * rows + t) * N;
    bool ok = DBG_REGION(o, N * sizeof(u64));
    for (uint32_t s = 0; s < S.n; s++)
        for (uint32_t j = 0; j < beta; j++)
            ok = ok && DBG_REGION(S.s[s].ext + (((size_t)b * beta + j) * rows + t) * N, N * sizeof(u64)) &&
                 DBG_REGION(S.s[s].key + ((size_t)(2 * j + pol) * (n_q + K) + pt) * N, N * sizeof(u64));
    if (!ok) return;
    const PrimeConst& pc = tb.pc[pt];
    const bool fp = pc.q < FESC_FP_LIMIT;
    const double q = pc.qd, qinv = pc.qinvd;
    const bool coef = last && t >= level;
    uint32_t n = 0, at[8];
    auto positions = [&](u64 g) {
#pragma unroll
        for (int e = 0; e < 8; e++) at[e] = g ? galois_src(tid + e * T, LOG, g) : tid + e * T;
    };
    auto put = [&](int e, u64 v) {
        if (coef) sm[at8<LOG, 1>(e)] = v;
        else o[tid + e * T] = v;
    };
    const size_t x_step = (size_t)rows * N, w_step = (size_t)2 * (n_q + K) * N;
    if (fp) {      // canonical words: products below 0.875 q, folded back every 7th (see k_inner)
        constexpr uint32_t G = 2;      // digits whose words are in flight together: a call of few ciphertexts is a chain of such waits
        double f[8];
#pragma unroll
        for (int e = 0; e < 8; e++) f[e] = accumulate ? fp_load(o[tid + e * T], q) : 0.0;
        for (uint32_t s = 0; s < S.n; s++) {
            const u64* x = S.s[s].ext + ((size_t)b * beta * rows + t) * N;
            const u64* w = S.s[s].key + ((size_t)pol * (n_q + K) + pt) * N + tid;
            positions(S.s[s].g);
            for (uint32_t j = 0; j < beta; j += G, x += G * x_step, w += G * w_step) {
                u64 xv[G][8], wv[G][8];
#pragma unroll
                for (uint32_t g = 0; g < G; g++)
                    if (j + g < beta) {
#pragma unroll
                        for (int e = 0; e < 8; e++) xv[g][e] = x[g * x_step + at[e]], wv[g][e] = __ldg(w + g * w_step + e * T);
                    }
#pragma unroll
                for (uint32_t g = 0; g < G; g++) {
                    if (j + g >= beta) break;
#pragma unroll
                    for (int e = 0; e < 8; e++) f[e] += fp_modmul(fp_from_u64(xv[g][e]), fp_from_u64(wv[g][e]), q, qinv);
                    if (n++ % 7 == 6) {
#pragma unroll
                        for (int e = 0; e < 8; e++) f[e] = fp_reduce(f[e], q, qinv);
                    }
                }
            }
        }
#pragma unroll
        for (int e = 0; e < 8; e++) put(e, fp_store(f[e], q, qinv));
    } else {
        acc128 a[8];
#pragma unroll
        for (int e = 0; e < 8; e++) a[e] = acc128{accumulate ? o[tid + e * T] : 0, 0};
        for (uint32_t s = 0; s < S.n; s++) {
            const u64* x = S.s[s].ext + ((size_t)b * beta * rows + t) * N;
            const u64* w = S.s[s].key + ((size_t)pol * (n_q + K) + pt) * N + tid;
            positions(S.s[s].g);
            for (uint32_t j = 0; j < beta; j++, x += x_step, w += w_step) {
                u64 xv[8], wv[8];
#pragma unroll
                for (int e = 0; e < 8; e++) xv[e] = x[at[e]], wv[e] = __ldg(w + e * T);
#pragma unroll
                for (int e = 0; e < 8; e++) mac128(a[e], xv[e], wv[e]);
                if (n++ % 8 == 7) {
#pragma unroll
                    for (int e = 0; e < 8; e++) a[e] = acc128{reduce128(a[e].hi, a[e].lo, pc), 0};
                }
            }
        }
#pragma unroll
        for (int e = 0; e < 8; e++) put(e, reduce128(a[e].hi, a[e].lo, pc));
    }
    if (!coef) return;
    __syncthreads();
    small_inv_row<LOG>(sm, tb, pt, scale + pt, o);
}
template <int LOG>
__global__ void __launch_bounds__(1 << (LOG - 3)) k_small_inner(InnerSrcs S, u64* acc, SmallTables tb, const InvScale* __restrict__ scale,
                                                                uint32_t level, uint32_t n_q, uint32_t K, uint32_t beta, int accumulate, int last) {
    const uint32_t t = blockIdx.x, pt = t < level ? t : n_q + (t - level);
    SMALL_BEGIN(last && t >= level, pt, true)
    inner_row<LOG>(sm, t, blockIdx.y, pt, blockIdx.z, S, acc, tb, scale, level, n_q, K, beta, accumulate, last);
}

// forward transform of v (canonical words), then out = (a - u) c (+ rot) (+ what out holds).  a and rot are a thread's words of the minuend
// and of the permuted c0 (zero: none), fetched by the caller before the transform needs its own.
struct SmallFinish {
    u64 cinv, cinvs;      // c and its Shoup companion
    int add;
};
template <int LOG>
__device__ __forceinline__ void small_words(u64 (&v)[8], const u64* p, u64 g) {      // words tid + k N/8 of the row p, through the permutation of g
    constexpr uint32_t T = (1u << LOG) / 8;
#pragma unroll
    for (int k = 0; k < 8; k++) {
        const uint32_t t = k * T + threadIdx.x;
        v[k] = !p ? 0 : p[g ? galois_src(t, LOG, g) : t];
    }
}
template <int LOG>
__device__ __forceinline__ void small_finish(u64 (&v)[8], u64* sm, const SmallTables& tb, uint32_t pi, const u64 (&a)[8], const u64 (&rot)[8], u64* out,
                                             const SmallFinish& fin) {
    constexpr uint32_t T = (1u << LOG) / 8;
    const uint32_t tid = threadIdx.x;
    const PrimeConst& pc = tb.pc[pi];
    if (pc.q < FESC_FP_LIMIT) {
        const FpS r{reinterpret_cast<const double*>(sm + SM_ROW(LOG)), pc.qd, pc.qinvd};
        double x[8];
#pragma unroll
        for (int k = 0; k < 8; k++) x[k] = fp_from_u64(v[k]);
        small_fwd<LOG>(r, x, sm);
        const double c = fp_from_u64(fin.cinv);
#pragma unroll
        for (int k = 0; k < 8; k++) {      // u is below 7.48q at the most (N = 2^11), a - u below 8q, the lazy product below 3.5q
            const uint32_t t = k * T + tid;
            double s = fp_modmul(fp_load(a[k], r.q) - FpS::value(sm[at8<LOG, 1>(k)]), c, r.q, r.qinv) + fp_load(rot[k], r.q);
            if (fin.add) s += fp_load(out[t], r.q);
            out[t] = fp_store(s, r.q, r.qinv);
        }
    } else {
        const IntS r{reinterpret_cast<const ulonglong2*>(sm + SM_ROW(LOG)), pc.q, 2 * pc.q};
        small_fwd<LOG>(r, v, sm);
#pragma unroll
        for (int k = 0; k < 8; k++) {
            const uint32_t t = k * T + tid;
            u64 s = addmod(shoup(submod(a[k], csub(csub(sm[at8<LOG, 1>(k)], r.q2), r.q), r.q), fin.cinv, fin.cinvs, r.q), rot[k], r.q);
            if (fin.add) s = addmod(s, out[t], r.q);
            out[t] = s;
        }
    }
}

// grid (level, 2, batch): out[b][p][i] = (acc[b][p][i] - u_i) P^-1 (+ ...), u_i = NTT(sum_k [y_k]_centred (P/p_k) mod q_i)
template <int LOG>
__device__ __forceinline__ void down_row(u64* sm, uint32_t i, uint32_t pol, uint32_t b, const u64* acc, u64* out, size_t out_stride,
                                         const ModDownTab* __restrict__ tab, const SmallTables& tb, uint32_t level, uint32_t K, int add_mask,
                                         const u64* rot_src, size_t rot_stride, u64 g) {
    constexpr uint32_t N = 1u << LOG, T = N / 8;
    const uint32_t tid = threadIdx.x;
    const u64* a = acc + ((size_t)b * 2 + pol) * (level + K) * N;
    u64* o = out + (size_t)b * out_stride + ((size_t)pol * level + i) * N;
    const u64* rot = rot_src && !pol ? rot_src + (size_t)b * rot_stride + (size_t)i * N : nullptr;
    if (!DBG_REGION(a, (size_t)(level + K) * N * sizeof(u64)) || !DBG_REGION(o, N * sizeof(u64)) || (rot && !DBG_REGION(rot, N * sizeof(u64)))) return;
    const PrimeConst& pc = tb.pc[i];
    const bool fp = pc.q < FESC_FP_LIMIT;
    const double q = pc.qd, qinv = pc.qinvd;
    u64 v[8], av[8], rv[8];
    small_words<LOG>(av, a + (size_t)i * N, 0);
    small_words<LOG>(rv, rot, g);
    const u64* src = a + (size_t)level * N + tid;
    if (fp) {
        double s[8];
#pragma unroll
        for (int k = 0; k < 8; k++) s[k] = 0.0;
        const double wrap = tab->wrapd[1][i], w = wrap + wrap >= q ? wrap - q : wrap;      // P, subtracted for every residue taken negative
        for (uint32_t m = 0; m < K; m++) {
            const u64 half = tab->half[m];
            const double m30 = tab->mat30d[m][i], m0 = tab->matd[m][i];
#pragma unroll
            for (int k = 0; k < 8; k++) {      // 30-bit halves: every product below 0.51 q, four times two of them and 4 w below 6.1 q
                const u64 y = src[(size_t)m * N + k * T];
                s[k] += fp_modmul(fp_from_u64(y >> 30), m30, q, qinv);
                s[k] += fp_modmul(fp_from_u64(y & ((1ull << 30) - 1)), m0, q, qinv);
                if (y > half) s[k] -= w;
                if (m == 3) s[k] = fp_reduce(s[k], q, qinv);
            }
        }
#pragma unroll
        for (int k = 0; k < 8; k++) v[k] = fp_store(s[k], q, qinv);
    } else {
#pragma unroll
        for (int k = 0; k < 8; k++) {
            acc128 w{0, 0};
            uint32_t n = 0;
            for (uint32_t m = 0; m < K; m++) {
                const u64 y = src[(size_t)m * N + k * T];
                n += y > tab->half[m];
                mac128(w, y, tab->mat[m][i]);
            }
            v[k] = submod(reduce128(w.hi, w.lo, pc), tab->wrap[n][i], pc.q);
        }
    }
    small_finish<LOG>(v, sm, tb, i, av, rv, o, SmallFinish{tab->pinv[i], tab->pinvs[i], (add_mask >> pol) & 1});
}
template <int LOG>
__global__ void __launch_bounds__(1 << (LOG - 3)) k_small_down(const u64* acc, u64* out, size_t out_stride, const ModDownTab* __restrict__ tab,
                                                               SmallTables tb, uint32_t level, uint32_t K, int add_mask, const u64* rot_src,
                                                               size_t rot_stride, u64 g) {
    SMALL_BEGIN(true, blockIdx.x, false)
    down_row<LOG>(sm, blockIdx.x, blockIdx.y, blockIdx.z, acc, out, out_stride, tab, tb, level, K, add_mask, rot_src, rot_stride, g);
}

// ---------------------------------------------------------------------------------------
// The four steps of a key switch with one key in one launch: a cluster of CTAs holds a ciphertext, its CTAs take the rows of a step in
// turn and meet at the cluster's barrier between steps (whose release and acquire also order the rows in global memory, so nothing
// written here is read through the read-only path).  The twiddle table of a CTA's first row of the next step is fetched while it waits.
// ---------------------------------------------------------------------------------------
struct SmallSwitch {
    const u64* src;              // the polynomial to be switched (k_small_coef)
    size_t src_stride;
    u64 *dcoef, *ext, *acc;
    int keep_own;
    u64 g;
    const u64* key;
    u64* out;
    size_t out_stride;
    int add_mask;
    const u64* rot_src;
    size_t rot_stride;
    const InvScale *up_scale, *down_scale;
    const ModUpDigit* up;
    const ModDownTab* down;
    uint32_t level, n_q, K, alpha, beta;
};
__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }

// grid (CTAs of a cluster, batch); 128 registers, so that an SM takes as many CTAs as the rule's figures were measured with
template <int LOG>
__global__ void __launch_bounds__(1 << (LOG - 3), 16 >> (LOG - 8)) k_small_switch(SmallSwitch a, SmallTables tb) {
    extern __shared__ __align__(16) u64 sm[];
    constexpr uint32_t N = 1u << LOG;
    const uint32_t rank = blockIdx.x, C = gridDim.x, b = blockIdx.y, level = a.level, rows = level + a.K, beta = a.beta, others = rows - a.alpha;
    const uint32_t n_up = beta * rows - level;
    // converted row `task`: every digit but the last has `others` of them (with one digit `others` may be anything)
    struct Up {
        uint32_t j, t, pt;
    };
    auto up_row = [&](uint32_t task) {
        Up u;
        u.j = beta == 1 ? 0 : task / others < beta - 1 ? task / others : beta - 1;
        const uint32_t d = u.j ? task - u.j * others : task, first = u.j * a.alpha, n = first + a.alpha < level ? a.alpha : level - first;
        u.t = d < first ? d : d + n;
        u.pt = u.t < level ? u.t : a.n_q + (u.t - level);
        return u;
    };
    if (rank < level) small_tables<LOG>(sm, tb, rank, true);
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    for (uint32_t l = rank; l < level; l += C) {
        if (l != rank) {
            __syncthreads();
            small_tables<LOG>(sm, tb, l, true);
        }
        coef_row<LOG>(sm, l, b, a.src, a.src_stride, a.keep_own ? a.ext : nullptr, (size_t)beta * rows * N, rows, a.alpha, a.dcoef, tb, a.up_scale, level, a.g);
    }
    __syncthreads();
    cluster_arrive();
    if (rank < n_up) small_tables<LOG>(sm, tb, up_row(rank).pt, false);
    cluster_wait();
    for (uint32_t task = rank; task < n_up; task += C) {
        const Up u = up_row(task);
        if (task != rank) {
            __syncthreads();
            small_tables<LOG>(sm, tb, u.pt, false);
        }
        modup_row<LOG>(sm, u.j, u.t, u.pt, b, a.dcoef, a.ext, a.up, tb, level, rows, beta);
    }
    __syncthreads();
    cluster_arrive();
    // the special rows first: they are transformed as well
    auto row_of = [&](uint32_t task) { return rows - 1 - (task >> 1); };
    if (rank < 2 * a.K) small_tables<LOG>(sm, tb, a.n_q + (row_of(rank) - level), true);
    cluster_wait();
    InnerSrcs S;
    S.n = 1;
    S.s[0] = InnerSrc{a.ext, a.key, 0};
    for (uint32_t task = rank; task < 2 * rows; task += C) {
        const uint32_t t = row_of(task), pt = t < level ? t : a.n_q + (t - level);
        if (task != rank && t >= level) {
            __syncthreads();
            small_tables<LOG>(sm, tb, pt, true);
        }
        inner_row<LOG>(sm, t, task & 1, pt, b, S, a.acc, tb, a.down_scale, level, a.n_q, a.K, beta, 0, 1);
    }
    __syncthreads();
    cluster_arrive();
    if (rank < 2 * level) small_tables<LOG>(sm, tb, rank >> 1, false);
    cluster_wait();
    for (uint32_t task = rank; task < 2 * level; task += C) {
        if (task != rank) {
            __syncthreads();
            small_tables<LOG>(sm, tb, task >> 1, false);
        }
        down_row<LOG>(sm, task >> 1, task & 1, b, a.acc, a.out, a.out_stride, a.down, tb, level, a.K, a.add_mask, a.rot_src, a.rot_stride, a.g);
    }
}

// grid (2, batch): COEFF form of the last limb of both polynomials to r[b][p]
template <int LOG>
__global__ void __launch_bounds__(1 << (LOG - 3)) k_small_last(const u64* in, size_t in_stride, u64* r, SmallTables tb, uint32_t level) {
    constexpr uint32_t N = 1u << LOG, T = N / 8;
    const uint32_t pol = blockIdx.x, b = blockIdx.y, tid = threadIdx.x;
    SMALL_BEGIN(true, level - 1, true)
    const u64* s = in + (size_t)b * in_stride + ((size_t)pol * level + level - 1) * N;
    u64* o = r + ((size_t)b * 2 + pol) * N;
    if (!DBG_REGION(s, N * sizeof(u64)) || !DBG_REGION(o, N * sizeof(u64))) return;
#pragma unroll
    for (int k = 0; k < 8; k++) sm[at8<LOG, 1>(k)] = s[k * T + tid];
    __syncthreads();
    small_inv_row<LOG>(sm, tb, level - 1, nullptr, o);
}
// grid (level - 1, 2, batch): out = (in - NTT(centred(r) mod q_i)) q_last^-1
template <int LOG>
__global__ void __launch_bounds__(1 << (LOG - 3), SM_CTAS(LOG)) k_small_rescale(const u64* in, size_t in_stride, const u64* r, u64* out,
                                                                  size_t out_stride, const RescaleTab* __restrict__ tab, SmallTables tb, uint32_t level) {
    constexpr uint32_t N = 1u << LOG, T = N / 8;
    const uint32_t i = blockIdx.x, pol = blockIdx.y, b = blockIdx.z, tid = threadIdx.x;
    SMALL_BEGIN(true, i, false)
    const u64* a = in + (size_t)b * in_stride + ((size_t)pol * level + i) * N;
    const u64* s = r + ((size_t)b * 2 + pol) * N;
    u64* o = out + (size_t)b * out_stride + ((size_t)pol * (level - 1) + i) * N;
    if (!DBG_REGION(a, N * sizeof(u64)) || !DBG_REGION(s, N * sizeof(u64)) || !DBG_REGION(o, N * sizeof(u64))) return;
    const PrimeConst& pc = tb.pc[i];
    u64 v[8], av[8], zero[8];
    small_words<LOG>(av, a, 0);
    small_words<LOG>(zero, nullptr, 0);
#pragma unroll
    for (int k = 0; k < 8; k++) {
        const u64 y = s[k * T + tid];
        u64 w = csub(y - mulhi(y, pc.mu) * pc.q, pc.q);
        if (y > tab->half) w = submod(w, tab->wrap[i], pc.q);
        v[k] = w;
    }
    small_finish<LOG>(v, sm, tb, i, av, zero, o, SmallFinish{tab->qinv[i], tab->qinvs[i], 0});
}

// ---------------------------------------------------------------------------------------
// launches
// ---------------------------------------------------------------------------------------
static cudaLaunchConfig_t cluster_config(uint32_t ctas, uint32_t batch, uint32_t threads, size_t smem, cudaStream_t st, cudaLaunchAttribute* attr) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(ctas, batch), cfg.blockDim = threads, cfg.dynamicSmemBytes = smem, cfg.stream = st;
    attr->id = cudaLaunchAttributeClusterDimension;
    attr->val.clusterDim.x = ctas, attr->val.clusterDim.y = attr->val.clusterDim.z = 1;
    cfg.attrs = attr, cfg.numAttrs = 1;
    return cfg;
}
template <int LOG>
static int small_attr(fesc_ctx* ctx) {
    const void* kernels[] = {(const void*)k_small_coef<LOG>, (const void*)k_small_modup<LOG>, (const void*)k_small_inner<LOG>, (const void*)k_small_down<LOG>,
                             (const void*)k_small_last<LOG>, (const void*)k_small_rescale<LOG>, (const void*)k_small_ntt<LOG, false>,
                             (const void*)k_small_ntt<LOG, true>, (const void*)k_small_switch<LOG>};
    for (const void* k : kernels) FESC_CHECK_CUDA(ctx, cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, SM_BYTES(LOG)));
    FESC_CHECK_CUDA(ctx, cudaFuncSetAttribute((const void*)k_small_switch<LOG>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1));
    for (int i = 0; i < 2; i++) {
        cudaLaunchAttribute attr;
        const cudaLaunchConfig_t cfg = cluster_config(8u << i, 1, 1u << (LOG - 3), SM_BYTES(LOG), 0, &attr);
        int n = 0;
        if (cudaOccupancyMaxActiveClusters(&n, k_small_switch<LOG>, &cfg) != cudaSuccess) cudaGetLastError(), n = 0;      // no cluster of this size
        ctx->small_clusters[i] = (uint32_t)n;
    }
    return FESC_OK;
}
int small_init(fesc_ctx* ctx) {      // up to 96 KB of shared memory per CTA
    return ctx->log_n == 12 ? small_attr<12>(ctx) : ctx->log_n == 11 ? small_attr<11>(ctx) : small_attr<10>(ctx);
}
bool small_ring(const fesc_ctx* ctx) { return ctx->log_n >= 10 && ctx->log_n <= 12; }
static SmallTables tables(const fesc_ctx* ctx) { return SmallTables{ctx->d_twf, ctx->d_itwf, ctx->d_tw, ctx->d_itw, ctx->d_pc}; }
#define SMALL_LAUNCH(kern, grid, ...)                                               \
    do {                                                                            \
        if (ctx->log_n == 12) launch(kern<12>, grid, 512, SM_BYTES(12), st, __VA_ARGS__);          \
        else if (ctx->log_n == 11) launch(kern<11>, grid, 256, SM_BYTES(11), st, __VA_ARGS__);     \
        else launch(kern<10>, grid, 128, SM_BYTES(10), st, __VA_ARGS__);                            \
        FESC_CHECK_CUDA(ctx, cudaGetLastError());                                   \
    } while (0)

int small_ntt_launch(fesc_ctx* ctx, u64* data, size_t rows, const RowMap& map, bool inverse, cudaStream_t st) {
    RowList l;
    l.period = map.period, l.count = 0;
    for (uint32_t i = 0; i < map.period; i++)
        if (map.prime[i] != 0xFF) l.row[l.count] = (uint8_t)i, l.prime[l.count++] = map.prime[i];
    const unsigned grid = (unsigned)(rows / map.period * l.count);
    if (!grid) return FESC_OK;
    const SmallTables tb = tables(ctx);
#define SMALL_NTT(LOG)                                                                              \
    do {                                                                                            \
        if (inverse) launch(k_small_ntt<LOG, true>, grid, 1 << (LOG - 3), SM_BYTES(LOG), st, data, tb, l);          \
        else launch(k_small_ntt<LOG, false>, grid, 1 << (LOG - 3), SM_BYTES(LOG), st, data, tb, l);                 \
    } while (0)
    if (ctx->log_n == 12) SMALL_NTT(12);
    else if (ctx->log_n == 11) SMALL_NTT(11);
    else SMALL_NTT(10);
#undef SMALL_NTT
    FESC_CHECK_CUDA(ctx, cudaGetLastError());
    return FESC_OK;
}

int small_decompose(fesc_ctx* ctx, const KsScratch& ws, const u64* src, size_t src_stride, bool keep_own, u64 g, uint32_t level, uint32_t batch,
                    cudaStream_t st) {
    const uint32_t beta = (level + ctx->alpha - 1) / ctx->alpha, rows = level + ctx->n_p;
    prof_begin(ctx, PF_NTT, st);
    SMALL_LAUNCH(k_small_coef, dim3(level, batch), src, src_stride, keep_own ? ws.ext : nullptr, (size_t)beta * rows * ctx->N, rows, ctx->alpha,
                 ws.dcoef, tables(ctx), ctx->tabs.d_up_scale + (size_t)(level - 1) * ctx->n_q, level, g);
    prof_end(ctx, PF_NTT, st);
    prof_begin(ctx, PF_MODUP, st);
    SMALL_LAUNCH(k_small_modup, dim3(beta * rows, batch), ws.dcoef, ws.ext, ctx->tabs.d_modup + (size_t)(level - 1) * ctx->beta_max, tables(ctx), level,
                 ctx->n_q, ctx->n_p, ctx->alpha, beta);
    prof_end(ctx, PF_MODUP, st);
    ctx->counters[0] += (uint64_t)batch * (level + beta * rows - level);
    return FESC_OK;
}
int small_inner(fesc_ctx* ctx, const KsScratch& ws, const InnerSrcs& S, uint32_t level, uint32_t batch, cudaStream_t st, int accumulate, int last) {
    const uint32_t beta = (level + ctx->alpha - 1) / ctx->alpha;
    prof_begin(ctx, PF_INNER, st);
    SMALL_LAUNCH(k_small_inner, dim3(level + ctx->n_p, 2, batch), S, ws.acc, tables(ctx), ctx->tabs.d_down_scale, level, ctx->n_q, ctx->n_p, beta,
                 accumulate, last);
    prof_end(ctx, PF_INNER, st);
    ctx->counters[1] += (uint64_t)batch * S.n;
    if (last) ctx->counters[0] += (uint64_t)batch * 2 * ctx->n_p;
    return FESC_OK;
}
int small_moddown(fesc_ctx* ctx, const KsScratch& ws, uint32_t level, uint32_t batch, u64* out, size_t out_stride, int add_mask, cudaStream_t st,
                  const u64* rot_src, size_t rot_stride, u64 g) {
    prof_begin(ctx, PF_MODDOWN, st);
    SMALL_LAUNCH(k_small_down, dim3(level, 2, batch), ws.acc, out, out_stride, ctx->tabs.d_moddown, tables(ctx), level, ctx->n_p, add_mask,
                 rot_src, rot_stride, g);
    prof_end(ctx, PF_MODDOWN, st);
    ctx->counters[0] += (uint64_t)batch * 2 * level;
    return FESC_OK;
}
int small_rescale(fesc_ctx* ctx, const u64* in, size_t in_stride, u64* out, size_t out_stride, uint32_t batch, uint32_t level, u64* r, cudaStream_t st) {
    prof_begin(ctx, PF_RESCALE, st);
    SMALL_LAUNCH(k_small_last, dim3(2, batch), in, in_stride, r, tables(ctx), level);
    SMALL_LAUNCH(k_small_rescale, dim3(level - 1, 2, batch), in, in_stride, r, out, out_stride, ctx->tabs.d_rescale + level, tables(ctx), level);
    prof_end(ctx, PF_RESCALE, st, 2);
    ctx->counters[0] += (uint64_t)batch * 2 * level;
    return FESC_OK;
}
// CTAs per ciphertext for one launch of k_small_switch, 0: the four kernels.  A barrier of a cluster costs less than a launch, but a step's rows are taken
// by the cluster's CTAs in turn: one launch while a CTA converts at most one row and the clusters leave a sixteenth of the device free (N = 2^10 / 2^11 /
// 2^12: 71 / 33 / 15 clusters of 8 and 31 / 14 / 7 of 16 fit; all 31 take 48 us where 28 take 30).  For five to eight rows both sizes will do: 16 while
// they are few.  One rotation each, four launches / 8 / 16 CTAs, us:
//   N = 2^12   3 limbs, 9 rows: 1 ciphertext 27.3 / 31.2 / 26.6, 6: 27.6 / 31.5 / 27.1, 15: 31.0 / 32.0 / -     4 limbs, 8 rows: 1: 38.2 / 41.0 / 38.8, 15: 51.7 / 41.6 / -
//              6 limbs, 18 rows: 1: 38.4 / 60.2 / 45.0       N = 2^11   2 limbs, 2 rows: 1: 27.7 / 28.9 / 28.7, 28: 36.8 / 32.6 / -
//   N = 2^11   4 limbs, 8 rows: 1: 28.4 / 31.0 / 29.3, 4: 30.9 / 31.5 / 29.8, 12: 36.9 / 31.7 / 33.6, 28: 43.9 / 35.9 / -     6 limbs, 18 rows: 8: 34.9 / 43.1 / 38.5
//   N = 2^10   4 limbs, 4 rows: 1: 31.1 / 29.0 / 27.3, 28: 38.0 / 30.6 / 32.6, 64: 49.2 / 34.0 / -     8 limbs, 16 rows: 1: 33.0 / 41.4 / 29.1, 28: 45.1 / 44.8 / 35.4
static uint32_t switch_ctas(const fesc_ctx* ctx, uint32_t level, uint32_t batch) {
    if (ctx->prof.on & (1u << PF_NTT | 1u << PF_MODUP | 1u << PF_INNER | 1u << PF_MODDOWN)) return 0;      // the steps are timed one by one
    const uint32_t beta = (level + ctx->alpha - 1) / ctx->alpha, n_up = beta * (level + ctx->n_p) - level;
    uint32_t most[2];      // clusters of 8 and of 16
    for (int i = 0; i < 2; i++) most[i] = ctx->small_clusters[i] - (ctx->small_clusters[i] + 15) / 16;
    if (n_up > (batch <= 6 ? 4 : 8) && n_up <= 16 && batch <= most[1]) return 16;
    if (n_up <= 8 && batch <= most[0]) return 8;
    return 0;
}
template <int LOG>
static int switch_launch(fesc_ctx* ctx, const SmallSwitch& a, uint32_t ctas, uint32_t batch, cudaStream_t st) {
    cudaLaunchAttribute attr[2];
    cudaLaunchConfig_t cfg = cluster_config(ctas, batch, 1u << (LOG - 3), SM_BYTES(LOG), st, attr);
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.numAttrs = 2;
    FESC_CHECK_CUDA(ctx, cudaLaunchKernelEx(&cfg, k_small_switch<LOG>, a, tables(ctx)));
    return FESC_OK;
}
bool small_switch(fesc_ctx* ctx, const KsScratch& ws, const u64* src, size_t src_stride, bool keep_own, u64 g, const u64* key, uint32_t level, uint32_t batch,
                  u64* out, size_t out_stride, int add_mask, cudaStream_t st, const u64* rot_src, size_t rot_stride, int& rc) {
    const uint32_t ctas = switch_ctas(ctx, level, batch), beta = (level + ctx->alpha - 1) / ctx->alpha, rows = level + ctx->n_p;
    if (!ctas) return false;
    const SmallSwitch a = {src, src_stride, ws.dcoef, ws.ext, ws.acc, keep_own, g, key, out, out_stride, add_mask, rot_src, rot_stride,
                           ctx->tabs.d_up_scale + (size_t)(level - 1) * ctx->n_q, ctx->tabs.d_down_scale, ctx->tabs.d_modup + (size_t)(level - 1) * ctx->beta_max,
                           ctx->tabs.d_moddown, level, ctx->n_q, ctx->n_p, ctx->alpha, beta};
    prof_begin(ctx, PF_NTT, st);
    rc = ctx->log_n == 12 ? switch_launch<12>(ctx, a, ctas, batch, st) : ctx->log_n == 11 ? switch_launch<11>(ctx, a, ctas, batch, st)
                                                                                          : switch_launch<10>(ctx, a, ctas, batch, st);
    if (rc != FESC_OK) return true;
    prof_end(ctx, PF_NTT, st);
    ctx->counters[0] += (uint64_t)batch * (beta * rows + 2 * ctx->n_p + 2 * level);
    ctx->counters[1] += batch;
    return true;
}

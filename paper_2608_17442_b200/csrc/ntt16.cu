// Negacyclic NTT / inverse NTT of N = 2^16 rows: two kernels of eight stages, 16 points per thread.
//
// Each kernel runs two register rounds of four stages and exchanges its points once, through shared memory:
//   * ntt16_cols: the stages with butterfly distance >= 256.  A CTA owns NTT_COLS adjacent columns of the 256 x 256 view.
//   * ntt16_rows: the stages with distance < 256.  A warp owns 512 adjacent points, so no CTA barrier is needed.
//
//   point index bits   15..12     11..8      7..4       3..0
//   round A            register   thread     (column)             stages 0..3 forward
//   round B            thread     register   (column)             stages 4..7
//   round C            (row)                 register   lane      stages 8..11
//   round D            (row)                 lane       register  stages 12..15
// The inverse runs D, C, B, A.
//
// What bounds it: a transform moves 2 MiB (0.32 us at the 6.55 TB/s a copy reaches) and issues about 17 cycles of FP64 work
// per warp-butterfly (0.26 us); measured 0.365 us per transform on 1536 rows, 0.41 on 384 (8 points per thread and two
// exchanges per kernel: 0.487 and 0.513).  Sixteen points per thread halve the shared-memory traffic and the barriers per
// butterfly and still fit 64 registers, i.e. 32 warps per SM; CTAs of four warps drift apart, so that loads, exchanges and
// butterflies of different CTAs overlap.  Measured beside it: 4 / 16 columns per CTA 0.432 / 0.372-0.381, 1 / 8 warps 0.397 /
// 0.387; one launch with the row in the shared memory of a cluster of 8 CTAs 0.54 (every seventh SM idle because a
// cluster needs 4 whole SMs of a GPC, barrier and store-release waits); launches split so that the second kernel finds its
// rows in L2 0.43-0.54 (launch tails).
#define FESC_DBG_FILE 11   // file id in the sites a debug build reports
#include "common.cuh"
#include "ntt16.cuh"

__device__ __forceinline__ uint32_t list_row(const RowList& list, uint32_t y, uint32_t& prime) {
    const uint32_t rep = y / list.count, e = y - rep * list.count;
    prime = list.prime[e];
    return rep * list.period + list.row[e];
}

// Constants of the primes that a kernel takes by value: none for integer rows (1 KB of parameters is 0.1 us of a
// launch: a rotation of one ciphertext of three 55-bit limbs 121.7 us with it, 120.5 without).
template <int A>
struct RowPrimes : PrimeDoubles {
    explicit RowPrimes(const fesc_ctx* ctx) : PrimeDoubles(ctx->pd) {}
};
template <>
struct RowPrimes<ROW_INT> {};

// grid = (256 / NTT_COLS, rows)
template <int A>
__global__ void __launch_bounds__(COL_THREADS, 1024 / COL_THREADS)
    ntt16_cols_fwd(u64* data, const void* __restrict__ tw, const PrimeConst* __restrict__ pcs, const __grid_constant__ RowPrimes<A> pd, RowList list,
                   uint32_t y0, int in_double, const u64* centred, double centred_q) {
    pdl_begin();
    __shared__ u64 sm[COL_SMEM(NTT_COLS)];
    uint32_t pi;
    const uint32_t row = list_row(list, y0 + blockIdx.y, pi);
    const uint32_t col = threadIdx.x % NTT_COLS, sub = threadIdx.x / NTT_COLS;
    if (!DBG_REGION(data + (size_t)row * N16, N16 * sizeof(u64))) return;      // the same for the whole CTA
    u64* p = data + (size_t)row * N16 + blockIdx.x * NTT_COLS + col;
    if constexpr (A == ROW_FP) {
        FpRow r{(const double*)tw + (size_t)pi * N16, pd.q[pi], pd.qinv[pi]};
        double x[16];
        if (centred) {                      // a row modulo another prime, centred, then folded modulo this one
            const u64* s = centred + (size_t)(row / list.period) * N16 + blockIdx.x * NTT_COLS + col;
            if (!DBG_REGION(centred + (size_t)(row / list.period) * N16, N16 * sizeof(u64))) return;
#pragma unroll
            for (int k = 0; k < 16; k++) x[k] = r.fold(fp_load(s[(16 * k + sub) * 256], centred_q));
        } else {
#pragma unroll
            for (int k = 0; k < 16; k++) {  // canonical words, or doubles with |x| <= q/2 from a conversion kernel
                const u64 v = ld_once(p + (16 * k + sub) * 256);
                x[k] = in_double ? FpRow::value(v) : fp_from_u64(v);
            }
        }
        fwd_cols<NTT_COLS, COLS_WORDS>(r, x, sm, col, sub, CtaBarrier());
#pragma unroll
        for (int k = 0; k < 16; k++) p[(16 * sub + k) * 256] = FpRow::bits(x[k]);      // doubles below 3.4q
    } else {
        const u64 q = pcs[pi].q;
        const IntRow r{(const ulonglong2*)tw + (size_t)pi * N16, q, 2 * q};
        u64 x[16];
#pragma unroll
        for (int k = 0; k < 16; k++) x[k] = p[(16 * k + sub) * 256];
        fwd_cols<NTT_COLS, COLS_WORDS>(r, x, sm, col, sub, CtaBarrier());
#pragma unroll
        for (int k = 0; k < 16; k++) p[(16 * sub + k) * 256] = x[k];                   // below 4q
    }
}

template <int A>
__global__ void __launch_bounds__(COL_THREADS, 1024 / COL_THREADS)
    ntt16_cols_inv(u64* data, const void* __restrict__ tw, const PrimeConst* __restrict__ pcs, const __grid_constant__ RowPrimes<A> pd, RowList list, uint32_t y0,
                   const InvScale* __restrict__ scale) {
    pdl_begin();
    __shared__ u64 sm[COL_SMEM(NTT_COLS)];
    uint32_t pi;
    const uint32_t row = list_row(list, y0 + blockIdx.y, pi);
    const uint32_t col = threadIdx.x % NTT_COLS, sub = threadIdx.x / NTT_COLS;
    if (!DBG_REGION(data + (size_t)row * N16, N16 * sizeof(u64))) return;
    u64* p = data + (size_t)row * N16 + blockIdx.x * NTT_COLS + col;
    const PrimeConst& pc = pcs[pi];
    if constexpr (A == ROW_FP) {
        FpRow r{(const double*)tw + (size_t)pi * N16, pd.q[pi], pd.qinv[pi]};
        double x[16];
#pragma unroll
        for (int k = 0; k < 16; k++) x[k] = FpRow::value(ld_once(p + (16 * sub + k) * 256));
        inv_cols<NTT_COLS>(r, x, sm, col, sub, CtaBarrier());
        const double ninv = scale ? scale[pi].nd : pc.ninvd, ninvw = scale ? scale[pi].wd : pc.ninvwd;
#pragma unroll
        for (int k = 0; k < 8; k++) {        // last stage, N^-1 folded in
            const double u = x[k], v = x[k + 8];
            p[(16 * k + sub) * 256] = fp_store(fp_modmul(u + v, ninv, r.q, r.qinv), r.q, r.qinv);
            p[(16 * (k + 8) + sub) * 256] = fp_store(fp_modmul(u - v, ninvw, r.q, r.qinv), r.q, r.qinv);
        }
    } else {
        const u64 q = pc.q;
        const IntRow r{(const ulonglong2*)tw + (size_t)pi * N16, q, 2 * q};
        u64 x[16];
#pragma unroll
        for (int k = 0; k < 16; k++) x[k] = p[(16 * sub + k) * 256];
        inv_cols<NTT_COLS>(r, x, sm, col, sub, CtaBarrier());
        const u64 n = scale ? scale[pi].n : pc.ninv, ns = scale ? scale[pi].ns : pc.ninvs;
        const u64 nw = scale ? scale[pi].w : pc.ninvw, nws = scale ? scale[pi].ws : pc.ninvws;
#pragma unroll
        for (int k = 0; k < 8; k++) {
            const u64 u = x[k], v = x[k + 8];
            p[(16 * k + sub) * 256] = shoup(u + v, n, ns, q);
            p[(16 * (k + 8) + sub) * 256] = shoup(u - v + r.q2, nw, nws, q);
        }
    }
}

// grid = (128 / NTT_WARPS, rows); FIN: the last step of a division instead of the plain store (NttFinish), 2: of a product
// WIDE: every buffer lies on a 16-byte boundary (a template and not a flag: tests of a flag at every access cost 0.4 % of a rotation)
template <int A, int FIN, bool WIDE>
__global__ void __launch_bounds__(ROW_THREADS, 1024 / ROW_THREADS)
    ntt16_rows_fwd(u64* data, const void* __restrict__ tw, const PrimeConst* __restrict__ pcs, const __grid_constant__ RowPrimes<A> pd, RowList list,
                   uint32_t y0, int out_double, NttFinish fin) {
    pdl_begin();
    __shared__ __align__(16) u64 sm_all[NTT_WARPS * ROW_SMEM];
    uint32_t pi;
    const uint32_t row = list_row(list, y0 + blockIdx.y, pi);
    const uint32_t lane = threadIdx.x & 31, warp = threadIdx.x >> 5, blk = blockIdx.x * NTT_WARPS + warp;
    u64* sm = sm_all + warp * ROW_SMEM;
    u64* p = data + (size_t)row * N16 + (size_t)blk * 512;
    if (!DBG_REGION(p, 512 * sizeof(u64))) return;      // warp barriers only
    const u64* in = p + 256 * (lane >> 4) + (lane & 15);
    const u64* s = sm + 2 * lane + 2 * (lane >> 3);     // the pair 2 lane (+ 64 j) of the padded buffer
    if constexpr (A == ROW_FP) {
        FpRow r{(const double*)tw + (size_t)pi * N16, pd.q[pi], pd.qinv[pi]};
        double x[16];
#pragma unroll
        for (int k = 0; k < 16; k++) x[k] = FpRow::value(ld_once(in + 16 * k));
        if (FIN) {
            const uint32_t bp = row / fin.level, i = row - bp * fin.level, ct = bp >> 1, pol = bp & 1, k = ct / fin.nb, b = ct - k * fin.nb;
            prefetch_l2(fin.acc + (size_t)ct * fin.acc_stride + ((size_t)pol * fin.acc_rows + i) * N16 + blk * 512 + 16 * lane);
            if (fin.rot_src && !pol)
                prefetch_l2(fin.rot_src + k * fin.rot_key_stride + b * fin.rot_stride + (size_t)i * N16 +
                            (galois_src(blk * 512, 16, fin.rot_g[k]) & ~511u) + 16 * lane);
        }
        fwd_rows<FIN != 0>(r, x, sm, blk, lane);
        const double q = r.q, qinv = r.qinv;
        if (!FIN) {
#pragma unroll
            for (int j = 0; j < 8; j++) {
                const ulonglong2 v = *reinterpret_cast<const ulonglong2*>(s + 72 * j);
                const double a = FpRow::value(v.x), b = FpRow::value(v.y);
                st_pair<WIDE>(p + 2 * lane + 64 * j, out_double ? make_ulonglong2(fp_handoff(a, q, qinv), fp_handoff(b, q, qinv))
                                                                : make_ulonglong2(fp_store(a, q, qinv), fp_store(b, q, qinv)));
            }
            return;
        }
        // (acc - u) c (+ sigma_g(c0)) (+ what the output holds); |acc - u| stays below 3.1q, the lazy product below 1.7q, the sum below 3.7q, so
        // every sum is exact and the words need not be centred first.  Rows of the buffer: row = bp * level + i.
        const uint32_t bp = row / fin.level, i = row - bp * fin.level, ct = bp >> 1, pol = bp & 1, kk = ct / fin.nb, b = ct - kk * fin.nb;
        const u64* acc = fin.acc + (size_t)ct * fin.acc_stride + ((size_t)pol * fin.acc_rows + i) * N16;
        u64* out = fin.out + kk * fin.out_key_stride + b * fin.out_stride + ((size_t)pol * fin.level + i) * N16;
        const u64* rot = fin.rot_src && !pol ? fin.rot_src + kk * fin.rot_key_stride + b * fin.rot_stride + (size_t)i * N16 : nullptr;
        const u64 rot_g = fin.rot_g[kk];
        if (!DBG_REGION(acc, N16 * sizeof(u64)) || !DBG_REGION(out, N16 * sizeof(u64)) || (rot && !DBG_REGION(rot, N16 * sizeof(u64)))) return;
        const double cinv = fin.cinv[i];
        const bool add = (fin.add_mask >> pol) & 1;
        // the registers of the transform are free: all eight minuends are requested at once, the other addends by fours
        const u64* pt = FIN == 2 && fin.pt ? fin.pt + ct * fin.pt_stride + (size_t)i * N16 + blk * 512 + 2 * lane : nullptr;
        if (pt && !DBG_REGION(pt - 2 * lane, 512 * sizeof(u64))) return;
        const double mul = FIN == 2 ? fp_mod_u64(fin.mul, pcs[pi]) : 0.0;
        ulonglong2 av[8];
#pragma unroll
        for (int j = 0; j < 8; j++) av[j] = ld_pair_once<WIDE>(acc + blk * 512 + 2 * lane + 64 * j);
#pragma unroll
        for (int h = 0; h < 8; h += 4) {
            ulonglong2 w[4];
            if (FIN == 1 && rot) {
#pragma unroll
                for (int j = 0; j < 4; j++) w[j] = galois_pair<WIDE>(rot, blk * 512 + 2 * lane + 64 * (h + j), 16, rot_g);
            }
#pragma unroll
            for (int j = h; j < h + 4; j++) {
                const ulonglong2 v = *reinterpret_cast<const ulonglong2*>(s + 72 * j);
                double a0 = fp_from_u64(av[j].x), a1 = fp_from_u64(av[j].y);
                if (FIN == 2) {             // lazy products below 0.875 q, the difference below 3 q
                    const ulonglong2 w2 = pt ? ld_pair_once<WIDE>(pt + 64 * j) : make_ulonglong2(0, 0);
                    a0 = fp_modmul(a0, pt ? fp_from_u64(w2.x) : mul, q, qinv);
                    a1 = fp_modmul(a1, pt ? fp_from_u64(w2.y) : mul, q, qinv);
                }
                double s0 = fp_modmul(a0 - FpRow::value(v.x), cinv, q, qinv);
                double s1 = fp_modmul(a1 - FpRow::value(v.y), cinv, q, qinv);
                if (FIN == 1 && rot) {
                    s0 += fp_from_u64(w[j - h].x);
                    s1 += fp_from_u64(w[j - h].y);
                }
                u64* o = out + blk * 512 + 2 * lane + 64 * j;
                if (FIN == 1 && add) {
                    const ulonglong2 ov = ld_pair_once<WIDE>(o);
                    s0 += fp_from_u64(ov.x);
                    s1 += fp_from_u64(ov.y);
                }
                st_pair_once<WIDE>(o, make_ulonglong2(fp_store(s0, q, qinv), fp_store(s1, q, qinv)));
            }
        }
    } else {
        const u64 q = pcs[pi].q;
        const IntRow r{(const ulonglong2*)tw + (size_t)pi * N16, q, 2 * q};
        u64 x[16];
#pragma unroll
        for (int k = 0; k < 16; k++) x[k] = ld_once(in + 16 * k);
        fwd_rows<false>(r, x, sm, blk, lane);
#pragma unroll
        for (int j = 0; j < 8; j++) {
            const ulonglong2 v = *reinterpret_cast<const ulonglong2*>(s + 72 * j);
            st_pair<WIDE>(p + 2 * lane + 64 * j, make_ulonglong2(r.canonical(v.x), r.canonical(v.y)));
        }
    }
}

template <int A, bool SRC, bool WIDE>
__global__ void __launch_bounds__(ROW_THREADS, 1024 / ROW_THREADS)
    ntt16_rows_inv(u64* data, const void* __restrict__ tw, const PrimeConst* __restrict__ pcs, const __grid_constant__ RowPrimes<A> pd, RowList list, uint32_t y0,
                   NttSource src) {
    pdl_begin();
    __shared__ __align__(16) u64 sm_all[NTT_WARPS * ROW_SMEM];
    uint32_t pi;
    const uint32_t row = list_row(list, y0 + blockIdx.y, pi);
    const uint32_t lane = threadIdx.x & 31, warp = threadIdx.x >> 5, blk = blockIdx.x * NTT_WARPS + warp;
    u64* sm = sm_all + warp * ROW_SMEM;
    u64* p = data + (size_t)row * N16 + (size_t)blk * 512;
    if (!DBG_REGION(p, 512 * sizeof(u64))) return;
    const u64* in = p + 2 * lane;
    uint32_t at = 0;                  // SRC: the words come from the permuted block that starts here
    u64* own = nullptr;
    const u64* pt = nullptr;
    u64 g = 0;
    if (SRC) {                        // rows of the buffer: row = polynomial * period + limb
        const uint32_t poly = row / list.period, l = row - poly * list.period, k = poly / src.nb, b = poly - k * src.nb;
        g = k < KS_MAX_KEYS ? src.g[k] : 0;
        in = src.src + k * src.key_stride + b * src.stride + (size_t)l * N16;
        if (src.own.ext) own = src.own.ext + own_index(src.own, poly, l, N16) + blk * 512 + 2 * lane;
        if (!DBG_REGION(in, N16 * sizeof(u64)) || (own && !DBG_REGION(own - 2 * lane, 512 * sizeof(u64)))) return;
        at = blk * 512 + 2 * lane;
        if (src.pt) {
            pt = src.pt + k * src.pt_stride + at;
            if (!DBG_REGION(pt - 2 * lane, 512 * sizeof(u64))) return;
        }
    }
    auto pair = [&](int j) {
        if (!SRC) return ld_pair<WIDE>(in + 64 * j);
        if (!g) return ld_pair<WIDE>(in + at + 64 * j);
        return galois_pair<WIDE>(in, at + 64 * j, 16, g);
    };
    u64* s = sm + 2 * lane + 2 * (lane >> 3);
    u64* o = p + 256 * (lane >> 4) + (lane & 15);
    if constexpr (A == ROW_FP) {
        FpRow r{(const double*)tw + (size_t)pi * N16, pd.q[pi], pd.qinv[pi]};
        const double mul = SRC ? fp_mod_u64(src.mul, pcs[pi]) : 0.0;
#pragma unroll
        for (int j = 0; j < 8; j++) {
            ulonglong2 v = pair(j);
            double a = fp_load(v.x, r.q), b = fp_load(v.y, r.q);
            if (SRC && (pt || src.mul)) {
                const ulonglong2 w = pt ? ld_pair<WIDE>(pt + 64 * j) : make_ulonglong2(0, 0);
                a = r.fold(fp_modmul(a, pt ? fp_from_u64(w.x) : mul, r.q, r.qinv));
                b = r.fold(fp_modmul(b, pt ? fp_from_u64(w.y) : mul, r.q, r.qinv));
            }
            v = make_ulonglong2(FpRow::bits(a), FpRow::bits(b));
            *reinterpret_cast<ulonglong2*>(s + 72 * j) = v;
            if (SRC && own) *reinterpret_cast<ulonglong2*>(own + 64 * j) = v;
        }
        __syncwarp();
        double x[16];
        inv_rows(r, x, sm, blk, lane);
#pragma unroll
        for (int k = 0; k < 16; k++) st_once(o + 16 * k, FpRow::bits(x[k]));      // doubles, |x| <= q/2
    } else {
        const u64 q = pcs[pi].q;
        const IntRow r{(const ulonglong2*)tw + (size_t)pi * N16, q, 2 * q};
#pragma unroll
        for (int j = 0; j < 8; j++) {
            const ulonglong2 v = pair(j);
            *reinterpret_cast<ulonglong2*>(s + 72 * j) = v;
            if (SRC && own) *reinterpret_cast<ulonglong2*>(own + 64 * j) = v;
        }
        __syncwarp();
        u64 x[16];
        inv_rows(r, x, sm, blk, lane);
#pragma unroll
        for (int k = 0; k < 16; k++) st_once(o + 16 * k, x[k]);                   // below 2q
    }
}

static bool all_aligned(const u64* data, const NttFinish& fin, const NttSource& src) {      // strides are multiples of N words
    const u64* all[] = {data, fin.acc, fin.out, fin.rot_src, fin.pt, src.src, src.pt};
    for (const u64* p : all)
        if (!pair_aligned(p)) return false;
    return true;
}
template <bool WIDE>
static int launch_all(fesc_ctx* ctx, u64* data, size_t rows, const RowMap& map, bool inverse, cudaStream_t st, bool in_double, bool out_double,
                      const NttFinish& fin, uint64_t& launches, const InvScale* scale, bool skip_cols, const NttSource* source) {
    RowList kind[2];
    for (RowList& l : kind) l.period = map.period, l.count = 0;
    for (uint32_t i = 0; i < map.period; i++) {
        if (map.prime[i] == 0xFF) continue;
        RowList& l = kind[ctx->q[map.prime[i]] < FESC_FP_LIMIT ? ROW_FP : ROW_INT];
        l.row[l.count] = (uint8_t)i;
        l.prime[l.count++] = map.prime[i];
    }
    const size_t reps = rows / map.period;
    const NttSource src = source ? *source : NttSource();
    for (int f = 0; f < 2; f++) {
        const RowList& l = kind[f];
        const size_t total = reps * l.count;
        for (size_t y0 = 0; y0 < total; y0 += 65535) {      // gridDim.y
            const unsigned n = (unsigned)(total - y0 < 65535 ? total - y0 : 65535);
            const dim3 gc(256 / NTT_COLS, n), gr(128 / NTT_WARPS, n);
            const uint32_t y = (uint32_t)y0;
            if (f == ROW_FP) {
                if (inverse) {
                    launch(source ? ntt16_rows_inv<ROW_FP, true, WIDE> : ntt16_rows_inv<ROW_FP, false, WIDE>, gr, ROW_THREADS, 0, st, data, ctx->d_itwf, ctx->d_pc, RowPrimes<ROW_FP>(ctx), l,
                           y, src);
                    if (!skip_cols) launch(ntt16_cols_inv<ROW_FP>, gc, COL_THREADS, 0, st, data, ctx->d_itwf, ctx->d_pc, RowPrimes<ROW_FP>(ctx), l, y, scale);
                } else {
                    if (!skip_cols) launch(ntt16_cols_fwd<ROW_FP>, gc, COL_THREADS, 0, st, data, ctx->d_twf, ctx->d_pc, RowPrimes<ROW_FP>(ctx), l, y, in_double, fin.centred, fin.centred_q);
                    if (fin.pt || fin.mul) launch(ntt16_rows_fwd<ROW_FP, 2, WIDE>, gr, ROW_THREADS, 0, st, data, ctx->d_twf, ctx->d_pc, RowPrimes<ROW_FP>(ctx), l, y, out_double, fin);
                    else if (fin.acc) launch(ntt16_rows_fwd<ROW_FP, 1, WIDE>, gr, ROW_THREADS, 0, st, data, ctx->d_twf, ctx->d_pc, RowPrimes<ROW_FP>(ctx), l, y, out_double, fin);
                    else launch(ntt16_rows_fwd<ROW_FP, 0, WIDE>, gr, ROW_THREADS, 0, st, data, ctx->d_twf, ctx->d_pc, RowPrimes<ROW_FP>(ctx), l, y, out_double, fin);
                }
            } else if (inverse) {
                launch(source ? ntt16_rows_inv<ROW_INT, true, WIDE> : ntt16_rows_inv<ROW_INT, false, WIDE>, gr, ROW_THREADS, 0, st, data, ctx->d_itw, ctx->d_pc, RowPrimes<ROW_INT>(), l, y,
                       src);
                if (!skip_cols) launch(ntt16_cols_inv<ROW_INT>, gc, COL_THREADS, 0, st, data, ctx->d_itw, ctx->d_pc, RowPrimes<ROW_INT>(), l, y, scale);
            } else {
                if (!skip_cols) launch(ntt16_cols_fwd<ROW_INT>, gc, COL_THREADS, 0, st, data, ctx->d_tw, ctx->d_pc, RowPrimes<ROW_INT>(), l, y, 0, nullptr, 0.0);
                launch(ntt16_rows_fwd<ROW_INT, 0, WIDE>, gr, ROW_THREADS, 0, st, data, ctx->d_tw, ctx->d_pc, RowPrimes<ROW_INT>(), l, y, 0, fin);
            }
            launches += skip_cols ? 1 : 2;
        }
    }
    return FESC_OK;
}

int ntt16_launch(fesc_ctx* ctx, u64* data, size_t rows, const RowMap& map, bool inverse, cudaStream_t st, bool in_double,
                 bool out_double, const NttFinish& fin, uint64_t& launches, const InvScale* scale, bool skip_cols, const NttSource* source) {
    const auto all = all_aligned(data, fin, source ? *source : NttSource()) ? launch_all<true> : launch_all<false>;
    return all(ctx, data, rows, map, inverse, st, in_double, out_double, fin, launches, scale, skip_cols, source);
}

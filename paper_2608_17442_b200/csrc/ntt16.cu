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
// per warp-butterfly (0.26 us); measured 0.383 us per transform on 1536 rows, 0.41 on 384 (8 points per thread and two
// exchanges per kernel: 0.487 and 0.513).  Sixteen points per thread halve the shared-memory traffic and the barriers per
// butterfly and still fit 64 registers, i.e. 32 warps per SM; CTAs of four warps drift apart, so that loads, exchanges and
// butterflies of different CTAs overlap.  Measured beside it: 4 / 16 columns per CTA 0.432 / 0.372-0.381, 1 / 8 warps 0.397 /
// 0.387; one launch with the row in the shared memory of a cluster of 8 CTAs 0.54 (every seventh SM idle because a
// cluster needs 4 whole SMs of a GPC, barrier and store-release waits); launches split so that the second kernel finds its
// rows in L2 0.43-0.54 (launch tails).
#define FESC_DBG_FILE 11   // file id in the sites a debug build reports
#include "common.cuh"
#include "ntt16.cuh"

#define N16 65536u
#ifndef NTT_COLS
#define NTT_COLS 8                  // columns per CTA of ntt16_cols (x 16 threads)
#endif
#ifndef NTT_WARPS
#define NTT_WARPS 4                 // warps per CTA of ntt16_rows
#endif
#define COL_THREADS (NTT_COLS * 16)
#define COL_SMEM (256 * NTT_COLS + 16 * 8)
#define ROW_THREADS (NTT_WARPS * 32)
#define ROW_SMEM 576                // words per warp: 512 points, two words of padding after every 16

__device__ __forceinline__ uint32_t pad16(uint32_t e) { return e + 2 * (e >> 4); }

// ---------------------------------------------------------------------------------------
// Arithmetic of a row.  w(i): twiddle i of the row's table.
// FpRow: primes below 2^50, exact products on the FP64 pipe.  |product| <= (1/2 + 1.5 |y| 2^-53) q with centred twiddles,
// so a forward stage takes a bound B q to (1.1875 B + 1/2) q: four stages from 2.8 q reach 8 q, seven from q/2 reach 7.88 q,
// and everything below 8 q < 2^53 is exact.  Forward rows are folded back to q/2 twice (after four and after eleven
// stages; the first bound leaves room for a conversion's lazy sum at the input); an inverse stage doubles the bound, so four stages from q/2 end at 8 q and every inverse
// round folds back.
// IntRow: any prime below 2^62, lazy Shoup butterflies, values below 4q (forward) or 2q (inverse).
// ---------------------------------------------------------------------------------------
struct FpRow {
    typedef double T;
    const double* __restrict__ tw;
    double q, qinv;
    __device__ __forceinline__ void ct(T& x, T& y, double w) const {
        const double v = fp_modmul(y, w, q, qinv), u = x;
        x = u + v;
        y = u - v;
    }
    __device__ __forceinline__ void gs(T& x, T& y, double w) const {
        const double u = x, v = y;
        x = u + v;
        y = fp_modmul(u - v, w, q, qinv);
    }
    template <int S>
    __device__ __forceinline__ void load(double (&w)[8], uint32_t i) const {      // 2^S twiddles from i on
        if (S == 0) {
            w[0] = __ldg(tw + i);
        } else {
#pragma unroll
            for (int k = 0; k < (1 << S) / 2; k++) {
                const double2 v = __ldg(reinterpret_cast<const double2*>(tw + i) + k);
                w[2 * k] = v.x, w[2 * k + 1] = v.y;
            }
        }
    }
    typedef double W;
    __device__ __forceinline__ T fold(T x) const { return fp_reduce(x, q, qinv); }
    static __device__ __forceinline__ u64 bits(T x) { return (u64)__double_as_longlong(x); }
    static __device__ __forceinline__ T value(u64 b) { return __longlong_as_double((long long)b); }
};
struct IntRow {
    typedef u64 T;
    typedef ulonglong2 W;
    const ulonglong2* __restrict__ tw;
    u64 q, q2;
    __device__ __forceinline__ void ct(T& x, T& y, const W& w) const {
        const u64 u = csub(x, q2), v = shoup_lazy(y, w.x, w.y, q);
        x = u + v;
        y = u - v + q2;
    }
    __device__ __forceinline__ void gs(T& x, T& y, const W& w) const {
        const u64 u = x, v = y;
        x = csub(u + v, q2);
        y = shoup_lazy(u - v + q2, w.x, w.y, q);
    }
    template <int S>
    __device__ __forceinline__ void load(W (&w)[8], uint32_t i) const {
#pragma unroll
        for (int k = 0; k < (1 << S); k++) w[k] = __ldg(tw + i + k);
    }
    __device__ __forceinline__ T fold(T x) const { return x; }
    static __device__ __forceinline__ u64 bits(T x) { return x; }
    static __device__ __forceinline__ T value(u64 b) { return b; }
};

// Stage S (0..3) of a forward round: distance 8 >> S, twiddles (i0 << S) + j for the j-th group of 16 >> S registers.
template <int S, class R>
__device__ __forceinline__ void fwd_stage(const R& r, typename R::T (&x)[16], uint32_t i0) {
    typename R::W w[8];
    r.template load<S>(w, i0 << S);
    constexpr int d = 8 >> S;
#pragma unroll
    for (int k = 0; k < 8; k++) {
        const int i = (k / d) * 2 * d + k % d;
        r.ct(x[i], x[i + d], w[k / d]);
    }
}
template <int S, class R>
__device__ __forceinline__ void inv_stage(const R& r, typename R::T (&x)[16], uint32_t i0) {
    typename R::W w[8];
    r.template load<S>(w, i0 << S);
    constexpr int d = 8 >> S;
#pragma unroll
    for (int k = 0; k < 8; k++) {
        const int i = (k / d) * 2 * d + k % d;
        r.gs(x[i], x[i + d], w[k / d]);
    }
}
template <class R>
__device__ __forceinline__ void fold16(const R& r, typename R::T (&x)[16]) {
#pragma unroll
    for (int k = 0; k < 16; k++) x[k] = r.fold(x[k]);
}

// position of (hi, col) in the exchange buffer of ntt16_cols: a row of 16 hi values is shifted by 8 words, so that both
// sides of the exchange are free of bank conflicts
__device__ __forceinline__ uint32_t col_slot(uint32_t hi, uint32_t col) { return hi * NTT_COLS + (hi >> 4) * 8 + col; }

// Rounds A and B on the registers of one thread (column, sub = 0..15).
template <class R>
__device__ __forceinline__ void fwd_cols(const R& r, typename R::T (&x)[16], u64* sm, uint32_t col, uint32_t sub) {
    fwd_stage<0>(r, x, 1);
    fwd_stage<1>(r, x, 1);
    fwd_stage<2>(r, x, 1);
    fwd_stage<3>(r, x, 1);
    fold16(r, x);
#pragma unroll
    for (int k = 0; k < 16; k++) sm[col_slot(16 * k, col) + sub * NTT_COLS] = R::bits(x[k]);
    __syncthreads();
    const u64* s = sm + col_slot(16 * sub, col);
#pragma unroll
    for (int k = 0; k < 16; k++) x[k] = R::value(s[k * NTT_COLS]);
    const uint32_t i0 = 16 + sub;
    fwd_stage<0>(r, x, i0);
    fwd_stage<1>(r, x, i0);
    fwd_stage<2>(r, x, i0);
    fwd_stage<3>(r, x, i0);
}
// Rounds B and A without the last stage.
template <class R>
__device__ __forceinline__ void inv_cols(const R& r, typename R::T (&x)[16], u64* sm, uint32_t col, uint32_t sub) {
    const uint32_t i0 = 16 + sub;
    inv_stage<3>(r, x, i0);
    inv_stage<2>(r, x, i0);
    inv_stage<1>(r, x, i0);
    inv_stage<0>(r, x, i0);
    fold16(r, x);
    u64* s = sm + col_slot(16 * sub, col);
#pragma unroll
    for (int k = 0; k < 16; k++) s[k * NTT_COLS] = R::bits(x[k]);
    __syncthreads();
#pragma unroll
    for (int k = 0; k < 16; k++) x[k] = R::value(sm[col_slot(16 * k, col) + sub * NTT_COLS]);
    inv_stage<3>(r, x, 1);
    inv_stage<2>(r, x, 1);
    inv_stage<1>(r, x, 1);
}
// Rounds C and D of one warp's 512 points (blk = index of the 512-point block in the row).  x holds round C's points on
// entry; on return the warp's padded buffer holds the transformed points, unreduced.
template <class R>
__device__ __forceinline__ void fwd_rows(const R& r, typename R::T (&x)[16], u64* sm, uint32_t blk, uint32_t lane) {
    const uint32_t i1 = 256 + 2 * blk + (lane >> 4);
    fwd_stage<0>(r, x, i1);
    fwd_stage<1>(r, x, i1);
    fwd_stage<2>(r, x, i1);
    fold16(r, x);
    fwd_stage<3>(r, x, i1);
    u64* c = sm + 288 * (lane >> 4) + (lane & 15);
#pragma unroll
    for (int k = 0; k < 16; k++) c[18 * k] = R::bits(x[k]);
    __syncwarp();
    ulonglong2* d = reinterpret_cast<ulonglong2*>(sm + 18 * lane);
#pragma unroll
    for (int k = 0; k < 8; k++) {
        const ulonglong2 v = d[k];
        x[2 * k] = R::value(v.x), x[2 * k + 1] = R::value(v.y);
    }
    const uint32_t i2 = 4096 + 32 * blk + lane;
    fwd_stage<0>(r, x, i2);
    fwd_stage<1>(r, x, i2);
    fwd_stage<2>(r, x, i2);
    fwd_stage<3>(r, x, i2);
#pragma unroll
    for (int k = 0; k < 8; k++) d[k] = make_ulonglong2(R::bits(x[2 * k]), R::bits(x[2 * k + 1]));
    __syncwarp();
}
// Rounds D and C: the warp's padded buffer holds the points on entry, x round C's points on return.
template <class R>
__device__ __forceinline__ void inv_rows(const R& r, typename R::T (&x)[16], u64* sm, uint32_t blk, uint32_t lane) {
    ulonglong2* d = reinterpret_cast<ulonglong2*>(sm + 18 * lane);
#pragma unroll
    for (int k = 0; k < 8; k++) {
        const ulonglong2 v = d[k];
        x[2 * k] = R::value(v.x), x[2 * k + 1] = R::value(v.y);
    }
    const uint32_t i2 = 4096 + 32 * blk + lane;
    inv_stage<3>(r, x, i2);
    inv_stage<2>(r, x, i2);
    inv_stage<1>(r, x, i2);
    inv_stage<0>(r, x, i2);
    fold16(r, x);
#pragma unroll
    for (int k = 0; k < 8; k++) d[k] = make_ulonglong2(R::bits(x[2 * k]), R::bits(x[2 * k + 1]));
    __syncwarp();
    const u64* c = sm + 288 * (lane >> 4) + (lane & 15);
#pragma unroll
    for (int k = 0; k < 16; k++) x[k] = R::value(c[18 * k]);
    const uint32_t i1 = 256 + 2 * blk + (lane >> 4);
    inv_stage<3>(r, x, i1);
    inv_stage<2>(r, x, i1);
    inv_stage<1>(r, x, i1);
    inv_stage<0>(r, x, i1);
    fold16(r, x);
}

__device__ __forceinline__ uint32_t list_row(const RowList& list, uint32_t y, uint32_t& prime) {
    const uint32_t rep = y / list.count, e = y - rep * list.count;
    prime = list.prime[e];
    return rep * list.period + list.row[e];
}

// grid = (256 / NTT_COLS, rows)
template <bool FP>
__global__ void __launch_bounds__(COL_THREADS, 1024 / COL_THREADS)
    ntt16_cols_fwd(u64* __restrict__ data, const void* __restrict__ tw, const PrimeConst* __restrict__ pcs, RowList list,
                   uint32_t y0, int in_double) {
    __shared__ u64 sm[COL_SMEM];
    uint32_t pi;
    const uint32_t row = list_row(list, y0 + blockIdx.y, pi);
    const uint32_t col = threadIdx.x % NTT_COLS, sub = threadIdx.x / NTT_COLS;
    if (!DBG_REGION(data + (size_t)row * N16, N16 * sizeof(u64))) return;      // the same for the whole CTA
    u64* p = data + (size_t)row * N16 + blockIdx.x * NTT_COLS + col;
    if (FP) {
        FpRow r{(const double*)tw + (size_t)pi * N16, pcs[pi].qd, pcs[pi].qinvd};
        double x[16];
#pragma unroll
        for (int k = 0; k < 16; k++) {      // canonical words, or doubles with |x| <= q/2 from a conversion kernel
            const u64 v = p[(16 * k + sub) * 256];
            x[k] = in_double ? FpRow::value(v) : fp_from_u64(v);
        }
        fwd_cols(r, x, sm, col, sub);
#pragma unroll
        for (int k = 0; k < 16; k++) p[(16 * sub + k) * 256] = FpRow::bits(x[k]);      // doubles below 3.7q
    } else {
        const u64 q = pcs[pi].q;
        IntRow r{(const ulonglong2*)tw + (size_t)pi * N16, q, 2 * q};
        u64 x[16];
#pragma unroll
        for (int k = 0; k < 16; k++) x[k] = p[(16 * k + sub) * 256];
        fwd_cols(r, x, sm, col, sub);
#pragma unroll
        for (int k = 0; k < 16; k++) p[(16 * sub + k) * 256] = x[k];                   // below 4q
    }
}

template <bool FP>
__global__ void __launch_bounds__(COL_THREADS, 1024 / COL_THREADS)
    ntt16_cols_inv(u64* __restrict__ data, const void* __restrict__ tw, const PrimeConst* __restrict__ pcs, RowList list, uint32_t y0) {
    __shared__ u64 sm[COL_SMEM];
    uint32_t pi;
    const uint32_t row = list_row(list, y0 + blockIdx.y, pi);
    const uint32_t col = threadIdx.x % NTT_COLS, sub = threadIdx.x / NTT_COLS;
    if (!DBG_REGION(data + (size_t)row * N16, N16 * sizeof(u64))) return;
    u64* p = data + (size_t)row * N16 + blockIdx.x * NTT_COLS + col;
    const PrimeConst& pc = pcs[pi];
    if (FP) {
        FpRow r{(const double*)tw + (size_t)pi * N16, pc.qd, pc.qinvd};
        double x[16];
#pragma unroll
        for (int k = 0; k < 16; k++) x[k] = FpRow::value(p[(16 * sub + k) * 256]);
        inv_cols(r, x, sm, col, sub);
        const double ninv = pc.ninvd, ninvw = pc.ninvwd;
#pragma unroll
        for (int k = 0; k < 8; k++) {        // last stage, N^-1 folded in
            const double u = x[k], v = x[k + 8];
            p[(16 * k + sub) * 256] = fp_store(fp_modmul(u + v, ninv, r.q, r.qinv), r.q, r.qinv);
            p[(16 * (k + 8) + sub) * 256] = fp_store(fp_modmul(u - v, ninvw, r.q, r.qinv), r.q, r.qinv);
        }
    } else {
        const u64 q = pc.q;
        IntRow r{(const ulonglong2*)tw + (size_t)pi * N16, q, 2 * q};
        u64 x[16];
#pragma unroll
        for (int k = 0; k < 16; k++) x[k] = p[(16 * sub + k) * 256];
        inv_cols(r, x, sm, col, sub);
        const u64 n = pc.ninv, ns = pc.ninvs, nw = pc.ninvw, nws = pc.ninvws;
#pragma unroll
        for (int k = 0; k < 8; k++) {
            const u64 u = x[k], v = x[k + 8];
            p[(16 * k + sub) * 256] = shoup(u + v, n, ns, q);
            p[(16 * (k + 8) + sub) * 256] = shoup(u - v + r.q2, nw, nws, q);
        }
    }
}

// grid = (128 / NTT_WARPS, rows); FIN: the last step of a division instead of the plain store (NttFinish)
template <bool FP, bool FIN>
__global__ void __launch_bounds__(ROW_THREADS, 1024 / ROW_THREADS)
    ntt16_rows_fwd(u64* __restrict__ data, const void* __restrict__ tw, const PrimeConst* __restrict__ pcs, RowList list,
                   uint32_t y0, int out_double, NttFinish fin) {
    __shared__ __align__(16) u64 sm_all[NTT_WARPS * ROW_SMEM];
    uint32_t pi;
    const uint32_t row = list_row(list, y0 + blockIdx.y, pi);
    const uint32_t lane = threadIdx.x & 31, warp = threadIdx.x >> 5, blk = blockIdx.x * NTT_WARPS + warp;
    u64* sm = sm_all + warp * ROW_SMEM;
    u64* p = data + (size_t)row * N16 + (size_t)blk * 512;
    if (!DBG_REGION(p, 512 * sizeof(u64))) return;      // warp barriers only
    const u64* in = p + 256 * (lane >> 4) + (lane & 15);
    const u64* s = sm + 2 * lane + 2 * (lane >> 3);     // the pair 2 lane (+ 64 j) of the padded buffer
    if (FP) {
        FpRow r{(const double*)tw + (size_t)pi * N16, pcs[pi].qd, pcs[pi].qinvd};
        double x[16];
#pragma unroll
        for (int k = 0; k < 16; k++) x[k] = FpRow::value(in[16 * k]);
        fwd_rows(r, x, sm, blk, lane);
        const double q = r.q, qinv = r.qinv;
        if (!FIN) {
            ulonglong2* o = reinterpret_cast<ulonglong2*>(p + 2 * lane);
#pragma unroll
            for (int j = 0; j < 8; j++) {
                const ulonglong2 v = *reinterpret_cast<const ulonglong2*>(s + 72 * j);
                const double a = FpRow::value(v.x), b = FpRow::value(v.y);
                o[32 * j] = out_double ? make_ulonglong2(fp_handoff(a, q, qinv), fp_handoff(b, q, qinv))
                                       : make_ulonglong2(fp_store(a, q, qinv), fp_store(b, q, qinv));
            }
            return;
        }
        // (acc - u) c (+ sigma_g(c0)) (+ what the output holds); |acc - u| stays below 5.4q, the lazy product below 1.6q, so
        // every sum is exact.  Rows of the buffer: row = bp * level + i.
        const uint32_t bp = row / fin.level, i = row - bp * fin.level, b = bp >> 1, pol = bp & 1;
        const u64* acc = fin.acc + (size_t)b * fin.acc_stride + ((size_t)pol * fin.acc_rows + i) * N16;
        u64* out = fin.out + (size_t)b * fin.out_stride + ((size_t)pol * fin.level + i) * N16;
        const u64* rot = fin.rot_src && !pol ? fin.rot_src + (size_t)b * fin.rot_stride + (size_t)i * N16 : nullptr;
        if (!DBG_REGION(acc, N16 * sizeof(u64)) || !DBG_REGION(out, N16 * sizeof(u64)) || (rot && !DBG_REGION(rot, N16 * sizeof(u64)))) return;
        const double cinv = fin.cinv[i];
        const bool add = (fin.add_mask >> pol) & 1;
#pragma unroll 4
        for (int j = 0; j < 8; j++) {
            const uint32_t t = blk * 512 + 2 * lane + 64 * j;
            const ulonglong2 v = *reinterpret_cast<const ulonglong2*>(s + 72 * j);
            const ulonglong2 av = *reinterpret_cast<const ulonglong2*>(acc + t);
            double s0 = fp_modmul(fp_load(av.x, q) - FpRow::value(v.x), cinv, q, qinv);
            double s1 = fp_modmul(fp_load(av.y, q) - FpRow::value(v.y), cinv, q, qinv);
            if (rot) {
                s0 += fp_load(rot[galois_src(t, 16, fin.rot_g)], q);
                s1 += fp_load(rot[galois_src(t + 1, 16, fin.rot_g)], q);
            }
            ulonglong2* o = reinterpret_cast<ulonglong2*>(out + t);
            if (add) {
                const ulonglong2 ov = *o;
                s0 += fp_load(ov.x, q);
                s1 += fp_load(ov.y, q);
            }
            *o = make_ulonglong2(fp_store(s0, q, qinv), fp_store(s1, q, qinv));
        }
    } else {
        const u64 q = pcs[pi].q;
        IntRow r{(const ulonglong2*)tw + (size_t)pi * N16, q, 2 * q};
        u64 x[16];
#pragma unroll
        for (int k = 0; k < 16; k++) x[k] = in[16 * k];
        fwd_rows(r, x, sm, blk, lane);
        ulonglong2* o = reinterpret_cast<ulonglong2*>(p + 2 * lane);
#pragma unroll
        for (int j = 0; j < 8; j++) {
            const ulonglong2 v = *reinterpret_cast<const ulonglong2*>(s + 72 * j);
            o[32 * j] = make_ulonglong2(csub(csub(v.x, r.q2), q), csub(csub(v.y, r.q2), q));
        }
    }
}

template <bool FP>
__global__ void __launch_bounds__(ROW_THREADS, 1024 / ROW_THREADS)
    ntt16_rows_inv(u64* __restrict__ data, const void* __restrict__ tw, const PrimeConst* __restrict__ pcs, RowList list, uint32_t y0) {
    __shared__ __align__(16) u64 sm_all[NTT_WARPS * ROW_SMEM];
    uint32_t pi;
    const uint32_t row = list_row(list, y0 + blockIdx.y, pi);
    const uint32_t lane = threadIdx.x & 31, warp = threadIdx.x >> 5, blk = blockIdx.x * NTT_WARPS + warp;
    u64* sm = sm_all + warp * ROW_SMEM;
    u64* p = data + (size_t)row * N16 + (size_t)blk * 512;
    if (!DBG_REGION(p, 512 * sizeof(u64))) return;
    const ulonglong2* in = reinterpret_cast<const ulonglong2*>(p + 2 * lane);
    u64* s = sm + 2 * lane + 2 * (lane >> 3);
    u64* o = p + 256 * (lane >> 4) + (lane & 15);
    if (FP) {
        FpRow r{(const double*)tw + (size_t)pi * N16, pcs[pi].qd, pcs[pi].qinvd};
#pragma unroll
        for (int j = 0; j < 8; j++) {
            const ulonglong2 v = in[32 * j];
            *reinterpret_cast<ulonglong2*>(s + 72 * j) = make_ulonglong2(FpRow::bits(fp_load(v.x, r.q)), FpRow::bits(fp_load(v.y, r.q)));
        }
        __syncwarp();
        double x[16];
        inv_rows(r, x, sm, blk, lane);
#pragma unroll
        for (int k = 0; k < 16; k++) o[16 * k] = FpRow::bits(x[k]);      // doubles, |x| <= q/2
    } else {
        const u64 q = pcs[pi].q;
        IntRow r{(const ulonglong2*)tw + (size_t)pi * N16, q, 2 * q};
#pragma unroll
        for (int j = 0; j < 8; j++) *reinterpret_cast<ulonglong2*>(s + 72 * j) = in[32 * j];
        __syncwarp();
        u64 x[16];
        inv_rows(r, x, sm, blk, lane);
#pragma unroll
        for (int k = 0; k < 16; k++) o[16 * k] = x[k];                   // below 2q
    }
}

int ntt16_launch(fesc_ctx* ctx, u64* data, size_t rows, const RowMap& map, bool inverse, cudaStream_t st, bool in_double,
                 bool out_double, const NttFinish& fin, uint64_t& launches) {
    RowList kind[2];                  // 0: primes below 2^50, 1: the rest
    for (RowList& l : kind) l.period = map.period, l.count = 0;
    for (uint32_t i = 0; i < map.period; i++) {
        if (map.prime[i] == 0xFF) continue;
        RowList& l = kind[ctx->q[map.prime[i]] < FESC_FP_LIMIT ? 0 : 1];
        l.row[l.count] = (uint8_t)i;
        l.prime[l.count++] = map.prime[i];
    }
    const size_t reps = rows / map.period;
    for (int f = 0; f < 2; f++) {
        const RowList& l = kind[f];
        const size_t total = reps * l.count;
        for (size_t y0 = 0; y0 < total; y0 += 65535) {      // gridDim.y
            const unsigned n = (unsigned)(total - y0 < 65535 ? total - y0 : 65535);
            const dim3 gc(256 / NTT_COLS, n), gr(128 / NTT_WARPS, n);
            const uint32_t y = (uint32_t)y0;
            if (f == 0 && !inverse) {
                ntt16_cols_fwd<true><<<gc, COL_THREADS, 0, st>>>(data, ctx->d_twf, ctx->d_pc, l, y, in_double);
                if (fin.acc) ntt16_rows_fwd<true, true><<<gr, ROW_THREADS, 0, st>>>(data, ctx->d_twf, ctx->d_pc, l, y, out_double, fin);
                else ntt16_rows_fwd<true, false><<<gr, ROW_THREADS, 0, st>>>(data, ctx->d_twf, ctx->d_pc, l, y, out_double, fin);
            } else if (f == 0) {
                ntt16_rows_inv<true><<<gr, ROW_THREADS, 0, st>>>(data, ctx->d_itwf, ctx->d_pc, l, y);
                ntt16_cols_inv<true><<<gc, COL_THREADS, 0, st>>>(data, ctx->d_itwf, ctx->d_pc, l, y);
            } else if (!inverse) {
                ntt16_cols_fwd<false><<<gc, COL_THREADS, 0, st>>>(data, ctx->d_tw, ctx->d_pc, l, y, 0);
                ntt16_rows_fwd<false, false><<<gr, ROW_THREADS, 0, st>>>(data, ctx->d_tw, ctx->d_pc, l, y, 0, fin);
            } else {
                ntt16_rows_inv<false><<<gr, ROW_THREADS, 0, st>>>(data, ctx->d_itw, ctx->d_pc, l, y);
                ntt16_cols_inv<false><<<gc, COL_THREADS, 0, st>>>(data, ctx->d_itw, ctx->d_pc, l, y);
            }
            launches += 2;
        }
    }
    return FESC_OK;
}

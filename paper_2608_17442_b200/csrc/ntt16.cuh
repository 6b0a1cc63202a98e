// Device code of the N = 2^16 transforms (ntt16.cu describes the decomposition) shared with the kernels that fuse one of
// their passes with a basis conversion.
#pragma once
#include "common.cuh"

// Row lists: the rows of one kind (arithmetic) inside a period of `period` rows.  Launch row y covers buffer row
// (y / count) * period + row[y % count] on prime[y % count].
struct RowList {
    uint32_t period, count;
    uint8_t row[252], prime[252];
};

#define N16 65536u
#ifndef NTT_COLS
#define NTT_COLS 8                  // columns per CTA of ntt16_cols (x 16 threads)
#endif
#ifndef NTT_WARPS
#define NTT_WARPS 4                 // warps per CTA of ntt16_rows
#endif
#define COL_THREADS (NTT_COLS * 16)
#define COL_SMEM(cols) (272 * (cols))
#define ROW_THREADS (NTT_WARPS * 32)
#define ROW_SMEM 576                // words per warp: 512 points, two words of padding after every 16

__device__ __forceinline__ uint32_t pad16(uint32_t e) { return e + 2 * (e >> 4); }

// ---------------------------------------------------------------------------------------
// Arithmetic of a row.  w(i): twiddle i of the row's table.
// FpRow: primes below 2^50, exact products on the FP64 pipe.  |product| <= (1/2 + 1.5 |y| 2^-53) q with centred twiddles,
// so a forward stage takes a bound B q to (1.1875 B + 1/2) q, and everything below 8 q < 2^53 is exact.  Where a bound would pass that, a stage
// folds the addends of its butterflies (half the points; the products reduce themselves) and leaves (1 + 0.1875 B) q.  Column pass of
// canonical words or words up to q: six stages to 7.62 q, folded at the seventh, 3.39 q; of converted words up to 2.51 q whose first stage has
// no products: 5.02, 6.47, folded at the third 2.22, 7.04 after the seventh, folded at the eighth 2.32 q; of words up to 0.7 q from the division by P
// likewise: 6.94 after the sixth, folded at the seventh, 3.24 q.  Row pass: 7.47 q at most after three stages, folded at the fourth 2.40, and
// 7.41 q at the end, or 2.10 q where the last stage folds as well.  An inverse stage doubles the bound, so four stages from q/2 end at 8 q and every
// inverse round folds back.
// IntRow: any prime below 2^62, lazy Shoup butterflies, values below 4q (forward) or 2q (inverse).
// ---------------------------------------------------------------------------------------
// SHARED: the twiddle table is a copy in shared memory.
template <bool SHARED, class V>
__device__ __forceinline__ V tw_load(const V* p) {
    return SHARED ? *p : __ldg(p);
}
template <bool SHARED>
struct FpRowT {
    typedef double T;
    const double* __restrict__ tw;
    double q, qinv;
    __device__ __forceinline__ void ct(T& x, T& y, double w) const {
        const double v = fp_modmul(y, w, q, qinv), u = x;
        x = u + v;
        y = u - v;
    }
    __device__ __forceinline__ void sums(T& x, T& y) const {       // a butterfly whose product is done
        const double u = x, v = y;
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
            w[0] = tw_load<SHARED>(tw + i);
        } else {
#pragma unroll
            for (int k = 0; k < (1 << S) / 2; k++) {
                const double2 v = tw_load<SHARED>(reinterpret_cast<const double2*>(tw + i) + k);
                w[2 * k] = v.x, w[2 * k + 1] = v.y;
            }
        }
    }
    template <int S>
    __device__ __forceinline__ void load_d(double (&w)[8], uint32_t blk, uint32_t lane) const {
        const double* t = tw + 4096 + 480 * blk;
        if (S == 0) {
            w[0] = tw_load<SHARED>(t + lane);
        } else {
            const double2* p = reinterpret_cast<const double2*>(t + 32) + 32 * ((1 << S) / 2 - 1) + lane;
#pragma unroll
            for (int k = 0; k < (1 << S) / 2; k++) {
                const double2 v = tw_load<SHARED>(p + 32 * k);
                w[2 * k] = v.x, w[2 * k + 1] = v.y;
            }
        }
    }
    __device__ __forceinline__ void one(double& w, uint32_t i) const { w = tw_load<SHARED>(tw + i); }
    typedef double W;
    __device__ __forceinline__ T fold(T x) const { return fp_reduce(x, q, qinv); }
    static __device__ __forceinline__ u64 bits(T x) { return (u64)__double_as_longlong(x); }
    static __device__ __forceinline__ T value(u64 b) { return __longlong_as_double((long long)b); }
};
typedef FpRowT<false> FpRow;
template <bool SHARED>
struct IntRowT {
    typedef u64 T;
    typedef ulonglong2 W;
    const ulonglong2* __restrict__ tw;
    u64 q, q2;
    __device__ __forceinline__ void ct(T& x, T& y, const W& w) const {
        const u64 u = csub(x, q2), v = shoup_lazy(y, w.x, w.y, q);
        x = u + v;
        y = u - v + q2;
    }
    __device__ __forceinline__ void sums(T& x, T& y) const {       // a butterfly whose product is done
        const u64 u = csub(x, q2), v = csub(y, q2);
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
        for (int k = 0; k < (1 << S); k++) w[k] = tw_load<SHARED>(tw + i + k);
    }
    template <int S>
    __device__ __forceinline__ void load_d(W (&w)[8], uint32_t blk, uint32_t lane) const {
        const ulonglong2* t = tw + 4096 + 480 * blk + lane;
#pragma unroll
        for (int k = 0; k < (1 << S); k++) w[k] = tw_load<SHARED>(t + 32 * ((1 << S) - 1 + k));
    }
    __device__ __forceinline__ void one(W& w, uint32_t i) const { w = tw_load<SHARED>(tw + i); }
    __device__ __forceinline__ u64 canonical(u64 x) const { return csub(csub(x, q2), q); }
    __device__ __forceinline__ T fold(T x) const { return x; }
    static __device__ __forceinline__ u64 bits(T x) { return x; }
    static __device__ __forceinline__ T value(u64 b) { return b; }
};
typedef IntRowT<false> IntRow;
// arithmetic of a launch's rows
enum { ROW_FP = 0, ROW_INT = 1 };

// Stage S (0..3) of a forward round: distance 8 >> S, twiddles (i0 << S) + j for the j-th group of 16 >> S registers.  FOLD: the addends are
// folded first.
template <int S, bool FOLD = false, class R>
__device__ __forceinline__ void fwd_stage(const R& r, typename R::T (&x)[16], uint32_t i0) {
    typename R::W w[8];
    r.template load<S>(w, i0 << S);
    constexpr int d = 8 >> S;
#pragma unroll
    for (int k = 0; k < 8; k++) {
        const int i = (k / d) * 2 * d + k % d;
        if (FOLD) x[i] = r.fold(x[i]);
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
// The same with the twiddles of round D: those of a 512-point block lie together, regrouped so that a warp's loads are
// contiguous (ntt16_twiddle_slot).
template <int S, bool FOLD = false, class R>
__device__ __forceinline__ void fwd_stage_d(const R& r, typename R::T (&x)[16], uint32_t blk, uint32_t lane) {
    typename R::W w[8];
    r.template load_d<S>(w, blk, lane);
    constexpr int d = 8 >> S;
#pragma unroll
    for (int k = 0; k < 8; k++) {
        const int i = (k / d) * 2 * d + k % d;
        if (FOLD) x[i] = r.fold(x[i]);
        r.ct(x[i], x[i + d], w[k / d]);
    }
}
template <int S, class R>
__device__ __forceinline__ void inv_stage_d(const R& r, typename R::T (&x)[16], uint32_t blk, uint32_t lane) {
    typename R::W w[8];
    r.template load_d<S>(w, blk, lane);
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

// position of (hi, col) in the exchange buffer of ntt16_cols: a row of 16 hi values is shifted by COLS words, so that both
// sides of the exchange are free of bank conflicts
template <int COLS>
__device__ __forceinline__ uint32_t col_slot(uint32_t hi, uint32_t col) { return hi * COLS + (hi >> 4) * COLS + col; }

__device__ __forceinline__ void prefetch_l2(const u64* p) { asm volatile("prefetch.global.L2 [%0];" ::"l"(p)); }
// all a transform needs of a context
struct SmallTables {
    const double *twf, *itwf;
    const ulonglong2 *tw, *itw;
    const PrimeConst* pc;
};
struct CtaBarrier {
    __device__ __forceinline__ void operator()() const { __syncthreads(); }
};
// What a column pass starts from: words up to q; converted words; words of the division by P.  The last two come with the products of the
// first stage done (their constants carry its twiddle) and share an exchange buffer that has been used before.
enum { COLS_WORDS, COLS_MODUP, COLS_MODDOWN };
// Rounds A and B on the registers of one thread (column, sub = 0..15); bar: barrier of the threads that share the columns.
template <int COLS, int FROM, class R, class B>
__device__ __forceinline__ void fwd_cols(const R& r, typename R::T (&x)[16], u64* sm, uint32_t col, uint32_t sub, B bar) {
    if (FROM == COLS_WORDS) {
        fwd_stage<0>(r, x, 1);
    } else {
#pragma unroll
        for (int k = 0; k < 8; k++) r.sums(x[k], x[k + 8]);
    }
    fwd_stage<1>(r, x, 1);
    fwd_stage<2, FROM == COLS_MODUP>(r, x, 1);
    fwd_stage<3>(r, x, 1);
    if (FROM != COLS_WORDS) bar();
#pragma unroll
    for (int k = 0; k < 16; k++) sm[col_slot<COLS>(16 * k, col) + sub * COLS] = R::bits(x[k]);
    bar();
    const u64* s = sm + col_slot<COLS>(16 * sub, col);
#pragma unroll
    for (int k = 0; k < 16; k++) x[k] = R::value(s[k * COLS]);
    const uint32_t i0 = 16 + sub;
    fwd_stage<0>(r, x, i0);
    fwd_stage<1>(r, x, i0);
    fwd_stage<2, FROM != COLS_MODUP>(r, x, i0);
    fwd_stage<3, FROM == COLS_MODUP>(r, x, i0);
}
// Rounds B and A without the last stage.
template <int COLS, class R, class B>
__device__ __forceinline__ void inv_cols(const R& r, typename R::T (&x)[16], u64* sm, uint32_t col, uint32_t sub, B bar) {
    const uint32_t i0 = 16 + sub;
    inv_stage<3>(r, x, i0);
    inv_stage<2>(r, x, i0);
    inv_stage<1>(r, x, i0);
    inv_stage<0>(r, x, i0);
    fold16(r, x);
    u64* s = sm + col_slot<COLS>(16 * sub, col);
#pragma unroll
    for (int k = 0; k < 16; k++) s[k * COLS] = R::bits(x[k]);
    bar();
#pragma unroll
    for (int k = 0; k < 16; k++) x[k] = R::value(sm[col_slot<COLS>(16 * k, col) + sub * COLS]);
    inv_stage<3>(r, x, 1);
    inv_stage<2>(r, x, 1);
    inv_stage<1>(r, x, 1);
}
// Rounds C and D of one warp's 512 points (blk = index of the 512-point block in the row).  x holds round C's points on
// entry; on return the warp's padded buffer holds the transformed points, unreduced (FOLD: the last stage folds).
template <bool FOLD, class R>
__device__ __forceinline__ void fwd_rows(const R& r, typename R::T (&x)[16], u64* sm, uint32_t blk, uint32_t lane) {
    const uint32_t i1 = 256 + 2 * blk + (lane >> 4);
    fwd_stage<0>(r, x, i1);
    fwd_stage<1>(r, x, i1);
    fwd_stage<2>(r, x, i1);
    fwd_stage<3, true>(r, x, i1);
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
    fwd_stage_d<0>(r, x, blk, lane);
    fwd_stage_d<1>(r, x, blk, lane);
    fwd_stage_d<2>(r, x, blk, lane);
    fwd_stage_d<3, FOLD>(r, x, blk, lane);
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
    inv_stage_d<3>(r, x, blk, lane);
    inv_stage_d<2>(r, x, blk, lane);
    inv_stage_d<1>(r, x, blk, lane);
    inv_stage_d<0>(r, x, blk, lane);
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

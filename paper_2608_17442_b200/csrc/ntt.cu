// Negacyclic NTT / inverse NTT over RNS limbs for sm_100a: rings N <= 2^9 and the entry point of all ring sizes
// (N = 2^16 lives in ntt16.cu, N = 2^10 .. 2^12 in small.cu).
//
// Forward: Cooley-Tukey butterflies with psi merged into the twiddles (natural order in, bit-reversed evaluation order
// out); inverse: Gentleman-Sande with the inverse twiddles and N^-1 folded into the last stage.
#define FESC_DBG_FILE 13   // file id in the sites a debug build reports
#include "common.cuh"

struct Tw {
    u64 w, s;
};
__device__ __forceinline__ Tw ldtw(const ulonglong2* __restrict__ t, uint32_t i) {
    ulonglong2 v = __ldg(t + i);
    return Tw{v.x, v.y};
}

// ---- classic lazy butterflies (any q < 2^62): forward values in [0,4q), inverse in [0,2q) ----
__device__ __forceinline__ void ct_bfly(u64& x, u64& y, const Tw& t, u64 q, u64 q2) {
    u64 u = csub(x, q2);
    u64 v = shoup_lazy(y, t.w, t.s, q);
    x = u + v;
    y = u - v + q2;
}
__device__ __forceinline__ void gs_bfly(u64& x, u64& y, const Tw& t, u64 q, u64 q2) {
    u64 u = x, v = y;
    x = csub(u + v, q2);
    y = shoup_lazy(u - v + q2, t.w, t.s, q);
}

// ---------------------------------------------------------------------------------------
// N <= 2^9: one CTA per row, radix-2 stages in shared memory.
// ---------------------------------------------------------------------------------------
template <bool INV>
__global__ void __launch_bounds__(256) ntt_small(u64* data, const ulonglong2* __restrict__ tw_all,
                                                 const PrimeConst* __restrict__ pcs, RowMap map, uint32_t log_n) {
    pdl_begin();
    const uint32_t row = blockIdx.x;
    const uint32_t pi = map.prime[row % map.period];
    if (pi == 0xFF) return;
    extern __shared__ u64 smx[];
    const uint32_t N = 1u << log_n;
    const PrimeConst pc = pcs[pi];
    const u64 q = pc.q, q2 = 2 * pc.q;
    const ulonglong2* tw = tw_all + (size_t)pi * N;
    u64* p = data + (size_t)row * N;
    if (!DBG_REGION(p, N * sizeof(u64)) || !DBG_REGION(tw, N * sizeof(ulonglong2))) return;
    for (uint32_t i = threadIdx.x; i < N; i += blockDim.x) smx[i] = p[i];
    __syncthreads();
    if (!INV) {
        for (uint32_t s = 0; s < log_n; s++) {
            const uint32_t t = N >> (s + 1);
            for (uint32_t b = threadIdx.x; b < N / 2; b += blockDim.x) {
                uint32_t i = b / t, k = b % t;
                uint32_t j = i * 2 * t + k;
                Tw w = ldtw(tw, (1u << s) + i);
                u64 x = smx[j], y = smx[j + t];
                ct_bfly(x, y, w, q, q2);
                smx[j] = x;
                smx[j + t] = y;
            }
            __syncthreads();
        }
        for (uint32_t i = threadIdx.x; i < N; i += blockDim.x) p[i] = csub(csub(smx[i], q2), q);
    } else {
        for (int s = (int)log_n - 1; s >= 1; s--) {
            const uint32_t t = N >> (s + 1);
            for (uint32_t b = threadIdx.x; b < N / 2; b += blockDim.x) {
                uint32_t i = b / t, k = b % t;
                uint32_t j = i * 2 * t + k;
                Tw w = ldtw(tw, (1u << s) + i);
                u64 x = smx[j], y = smx[j + t];
                gs_bfly(x, y, w, q, q2);
                smx[j] = x;
                smx[j + t] = y;
            }
            __syncthreads();
        }
        const uint32_t t = N / 2;
        for (uint32_t b = threadIdx.x; b < N / 2; b += blockDim.x) {
            u64 u = smx[b], v = smx[b + t];
            p[b] = shoup(u + v, pc.ninv, pc.ninvs, q);
            p[b + t] = shoup(u - v + q2, pc.ninvw, pc.ninvws, q);
        }
    }
}

int ntt_launch(fesc_ctx* ctx, u64* d_data, size_t rows, const RowMap& map, bool inverse, cudaStream_t st, bool in_double,
               bool out_double, const NttFinish* finish, const InvScale* scale, bool skip_cols, const NttSource* source) {
    const NttFinish fin = finish ? *finish : NttFinish();
    if (fin.acc && (inverse || ctx->log_n != 16)) return fesc_fail(ctx, FESC_EINVAL, "ntt: the fused epilogue belongs to a forward N = 2^16 transform");
    if ((scale || skip_cols || source) && ctx->log_n != 16) return fesc_fail(ctx, FESC_EINVAL, "ntt: N = 2^16 only");
    if (rows == 0) return FESC_OK;
    if (rows > 0x7fffffffu) return fesc_fail(ctx, FESC_EINVAL, "ntt: too many rows");
    const ulonglong2* tw = inverse ? ctx->d_itw : ctx->d_tw;
    size_t live = 0;
    for (uint32_t i = 0; i < map.period; i++) live += map.prime[i] != 0xFF;
    ctx->counters[0] += rows / map.period * live;
    ctx->counters[6] += rows / map.period * live * (skip_cols ? 1 : 2);
    prof_begin(ctx, PF_NTT, st);
    uint64_t launches = 0;
    if (ctx->log_n == 16) {
        const int rc = ntt16_launch(ctx, d_data, rows, map, inverse, st, in_double, out_double, fin, launches, scale, skip_cols, source);
        if (rc != FESC_OK) return rc;
    } else if (small_ring(ctx)) {
        const int rc = small_ntt_launch(ctx, d_data, rows, map, inverse, st);
        if (rc != FESC_OK) return rc;
        launches = 1;
    } else {
        size_t smem = sizeof(u64) << ctx->log_n;
        if (!inverse)
            launch(ntt_small<false>, (unsigned)rows, 256, smem, st, d_data, tw, ctx->d_pc, map, ctx->log_n);
        else
            launch(ntt_small<true>, (unsigned)rows, 256, smem, st, d_data, tw, ctx->d_pc, map, ctx->log_n);
        launches = 1;
    }
    prof_end(ctx, PF_NTT, st, launches);
    FESC_CHECK_CUDA(ctx, cudaGetLastError());
    return FESC_OK;
}

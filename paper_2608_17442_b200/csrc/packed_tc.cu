// BSGS accumulate for periodic diagonals on the fifth-generation tensor cores (tcgen05).
//
// Periodic diagonals hold one image per aligned run of 2^dshift coefficients, so the products of a run share their left operand:
// for 128 (b,p) outputs it is 128 rows x 7 byte planes x at most 192 terms, 168 KB, and stays in shared memory while the inputs of
// the run's coefficients (4 token blocks x 2 polynomials x 7 planes, 10.5 KB each) stream past it.  The kernel for diagonals that
// differ at every coefficient (packed.cu) has to fetch both operands of every product and recombine 49 sums in registers; on periodic
// images its tensor pipe was 0.62 busy and is several times narrower.
//
// One instruction multiplies byte plane k of the 128 outputs with all planes j of the inputs, and the sums of equal weight 256^(k+j)
// belong together.  Those of planes 2m and 2m + 1 land together: both have the accumulator m of eight column groups, plane 2m + 1 takes its
// inputs from one group early, where a group of zeros lies, so that column group y holds the weight 256^(2m + y).  A thread owns an output:
// it adds the groups of equal weight of the four accumulators, and no exchange between lanes is left.  64 columns per instruction.
//
// Two tcgen05.mma are ordered without a wait between them only when they have the same accumulator and the same shape.  Products that
// depend on one another therefore share both, and the accumulators share no column; all of tensor memory is taken (2 x 4 x 64).
//
// 8 token blocks of 210 outputs x 189 terms at 6 limbs: 20.1 ms (40.8 ms in packed.cu).  With accumulators that overlap, so that the 13 sums
// are read without an addition, 19.6, but on an order that nothing promises; two accumulators of four planes in 80 columns 21.1, one of seven in 112
// columns 22.8; the products in other orders 20.3.  An instruction of 128 x 64 x 32 takes 48 cycles, what reading its operands from shared memory
// takes, so the products alone need 11.5 ms; outputs are scattered sectors.
//
// CTA = 10 warps: 8 recombine (thread = output and half of the columns), one issues the products, one fetches the inputs.  Two sets of accumulators (2 x 256 columns of
// tensor memory) let the recombination of a coefficient run beside the products of the next.  Every wait is bounded (status word 4).
#define FESC_DBG_FILE 15   // file id in the sites a debug build reports
#include "ops.cuh"

#define TC_FRAG 1792                       // bytes of one coefficient's inputs per k-step of 32 terms: [plane][k half][8 rows][16]
#define TC_CORE 256                        // 8 rows x 32 terms: two core matrices of 8 x 16 bytes
#define TC_MAX_KSTEPS 6
#define TC_THREADS 320
#define TC_OUT_WARPS 8
#define TC_BUFFERS 4
#define TC_A_BYTES(ksteps) (7u * (ksteps) * 16 * TC_CORE)
#define TC_PLANES 2                        // byte planes of the outputs per accumulator
#define TC_ACCS ((7 + TC_PLANES - 1) / TC_PLANES)
#define TC_GROUPS ((7 + TC_PLANES) / 2 * 2)                      // 7 + TC_PLANES - 1 column groups of 8, made even (columns come in 16s)
#define TC_GAP (TC_GROUPS - 7)                                   // groups of zeros before and after every k-step's seven planes
#define TC_ACC_COLS (256 / TC_ACCS / 32 * 32)                    // columns of tensor memory from one accumulator to the next
#define TC_B_BYTES(ksteps) ((TC_GAP + (7u + TC_GAP) * (ksteps)) * TC_CORE)
static_assert(8 * TC_GROUPS <= TC_ACC_COLS && TC_ACCS * TC_ACC_COLS <= 256, "accumulators do not share columns");
static_assert(TC_PLANES - 1 <= TC_GAP, "a window starts at most TC_PLANES - 1 groups early");

// Shared-memory operand without swizzle, both core matrices of a row group side by side: K direction 128 bytes, row groups 256.  Only the
// address, in the low word, differs between operands: one thread issues all products, and what it computes per product counts.
#define TC_DESC_HI ((uint32_t)(TC_CORE >> 4) | (1u << 14))
__device__ __forceinline__ uint32_t tc_desc(uint32_t addr) { return (addr >> 4) | ((uint32_t)(128 >> 4) << 16); }
__device__ __forceinline__ void tc_mma(uint32_t d, uint32_t a, uint32_t b, uint32_t idesc, bool add) {
    asm volatile("{\n\t.reg .pred p;\n\t.reg .b64 a, b;\n\tmov.b64 a, {%1, %5};\n\tmov.b64 b, {%2, %5};\n\tsetp.ne.u32 p, %4, 0;\n\t"
                 "tcgen05.mma.cta_group::1.kind::i8 [%0], a, b, %3, p;\n\t}" ::"r"(d), "r"(a), "r"(b), "r"(idesc), "r"((uint32_t)add), "r"(TC_DESC_HI)
                 : "memory");
}
__device__ __forceinline__ void tc_commit(uint32_t bar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void tc_ld4(uint32_t* r, uint32_t addr) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0, %1, %2, %3}, [%4];" : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr));
}

// column groups of accumulator a that hold sums: its planes plus the seven of the inputs, less one
__host__ __device__ constexpr int tc_groups(int a) { return (7 - TC_PLANES * a < TC_PLANES ? 7 - TC_PLANES * a : TC_PLANES) + 6; }

template <bool FP, int KS>
__global__ void __launch_bounds__(TC_THREADS, 1)
    k_bsgs_accumulate_periodic(const uint8_t* __restrict__ xpk, const uint8_t* __restrict__ dpk, u64* __restrict__ acc,
                               const PrimeConst* __restrict__ pcs, uint32_t N, uint32_t level, uint32_t tbs, uint32_t bp_count, uint32_t dshift,
                               uint32_t buffers, uint32_t* __restrict__ status) {
    constexpr uint32_t ksteps = KS;
    extern __shared__ __align__(128) uint8_t smem[];
    __shared__ __align__(8) u64 bars[2 * TC_BUFFERS + 5];
    __shared__ uint32_t tmem_base;
    const uint32_t tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    // the CTAs that share a run's operands are neighbours in the grid and share them through L2
    const uint32_t tbts = (tbs + 3) >> 2, mts = (bp_count + 127) >> 7, l = blockIdx.y;
    const uint32_t mt = blockIdx.x % mts, tbt = blockIdx.x / mts % tbts, run = blockIdx.x / (mts * tbts);
    const uint32_t tiles = N >> 3, tiles_d = tiles >> dshift, bp_tiles = (bp_count + 7) >> 3, coefs = 1u << dshift, c_first = run << dshift;
    const size_t stage = 8 * TC_FRAG, poly = (size_t)level * N, ctw = 2 * poly;
    const uint8_t* dsrc = dpk + ((size_t)l * tiles_d + (run >> 3)) * ksteps * stage + (run & 7) * TC_FRAG;
    const size_t tile_stride = (size_t)level * tiles_d * ksteps * stage;
    const uint8_t* xsrc = xpk + ((size_t)tbt * level + l) * tiles * ksteps * stage;
#ifdef FESC_DEBUG_BOUNDS
    {   // the same outcome for every thread of the CTA (barriers follow)
        bool ok = DBG_REGION(xsrc + (size_t)(c_first >> 3) * ksteps * stage, ((size_t)((c_first + coefs - 1) >> 3) - (c_first >> 3) + 1) * ksteps * stage);
        for (uint32_t bt = mt * 16; bt < mt * 16 + 16 && bt < bp_tiles && ok; bt++)
            ok = DBG_REGION(dsrc + bt * tile_stride, (size_t)(ksteps - 1) * stage + TC_FRAG);
        for (uint32_t tb = tbt * 4; tb < tbt * 4 + 4 && tb < tbs && ok; tb++)
            ok = DBG_REGION(acc + (size_t)tb * bp_count * ctw, (size_t)bp_count * ctw * sizeof(u64));
        if (!ok) return;
    }
#endif
    const uint32_t a_base = (uint32_t)__cvta_generic_to_shared(smem), a_bytes = TC_A_BYTES(ksteps), b_bytes = TC_B_BYTES(ksteps);
    const uint32_t b_base = a_base + a_bytes, bar = (uint32_t)__cvta_generic_to_shared(bars);
    const uint32_t b_full = bar, b_free = bar + 8 * TC_BUFFERS, d_full = bar + 16 * TC_BUFFERS, d_free = d_full + 16, drained = d_free + 16;
    if (warp == TC_OUT_WARPS) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 512;" ::"r"((uint32_t)__cvta_generic_to_shared(&tmem_base))
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    if (tid == 0) {
        for (uint32_t i = 0; i < TC_BUFFERS; i++) mbar_init(b_full + 8 * i, 1), mbar_init(b_free + 8 * i, 1);
        for (uint32_t i = 0; i < 2; i++) mbar_init(d_full + 8 * i, 1), mbar_init(d_free + 8 * i, TC_OUT_WARPS);
        mbar_init(drained, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    // zeros around the inputs, and the left operand: [k-step][plane][16 row groups][k half][8 rows][16 bytes]
    for (uint32_t i = tid; i < buffers * b_bytes / 16; i += TC_THREADS) *reinterpret_cast<uint4*>(smem + a_bytes + 16 * i) = make_uint4(0, 0, 0, 0);
    for (uint32_t i = warp; i < 16 * ksteps; i += TC_THREADS / 32) {
        const uint32_t rg = i / ksteps, ks = i - rg * ksteps, bt = mt * 16 + rg;
        uint32_t lo[7] = {}, hi[7] = {};
        if (bt < bp_tiles) {
            const uint8_t* img = dsrc + bt * tile_stride + ks * stage;
#pragma unroll
            for (int m = 0; m < 3; m++) {
                const uint4 v = __ldg(reinterpret_cast<const uint4*>(img + 512 * m) + lane);
                lo[2 * m] = v.x, lo[2 * m + 1] = v.y, hi[2 * m] = v.z, hi[2 * m + 1] = v.w;
            }
            const uint2 v = __ldg(reinterpret_cast<const uint2*>(img + 1536) + lane);
            lo[6] = v.x, hi[6] = v.y;
        }
#pragma unroll
        for (int p = 0; p < 7; p++) {
            uint32_t* dst = reinterpret_cast<uint32_t*>(smem + ((ks * 7 + p) * 16 + rg) * TC_CORE) + lane;
            dst[0] = lo[p], dst[32] = hi[p];
        }
    }
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = tmem_base;
    bool ok = true;
    if (warp == TC_OUT_WARPS + 1) {                       // fetches the inputs
        if (lane == 0) {
            uint32_t i = 0;
            for (; i < coefs; i++) {
                const uint32_t buf = i % buffers, use = i / buffers, c = c_first + i;
                if (use && mbar_wait_bounded(b_free + 8 * buf, (use - 1) & 1)) {
                    ok = false;
                    break;
                }
                const uint8_t* src = xsrc + (size_t)(c >> 3) * ksteps * stage + (c & 7) * TC_FRAG;
                mbar_expect_tx(b_full + 8 * buf, ksteps * TC_FRAG);
                for (uint32_t k = 0; k < ksteps; k++)
                    bulk_g2s(b_base + buf * b_bytes + (TC_GAP + (7 + TC_GAP) * k) * TC_CORE, src + k * stage, TC_FRAG, b_full + 8 * buf);
            }
            // copies in flight when a wait ran out: the last `buffers` of them
            if (!ok)
                for (uint32_t s = i > buffers ? i - buffers : 0; s < i; s++) mbar_wait_bounded(b_full + 8 * (s % buffers), (s / buffers) & 1);
        }
    } else if (warp == TC_OUT_WARPS) {                // issues the products
        if (lane == 0) {
            // u8 x u8 -> s32, both operands K-major, 128 rows
            const uint32_t idesc = (2u << 4) | (TC_GROUPS << 17) | (8u << 24), a0 = tc_desc(a_base);
            for (uint32_t i = 0; i < coefs; i++) {
                const uint32_t buf = i % buffers, use = i / buffers, db = i & 1, du = i >> 1;
                if (mbar_wait_bounded(b_full + 8 * buf, use & 1) || (du && mbar_wait_bounded(d_free + 8 * db, (du - 1) & 1))) {
                    ok = false;
                    break;
                }
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                const uint32_t b0 = tc_desc(b_base + TC_GAP * TC_CORE + buf * b_bytes), d = tmem + 256 * db;
#pragma unroll
                for (uint32_t k = 0; k < KS; k++)
#pragma unroll
                    for (uint32_t p = 0; p < 7; p++)
                        tc_mma(d + TC_ACC_COLS * (p / TC_PLANES), a0 + (k * 7 + p) * TC_CORE,
                               b0 + ((7 + TC_GAP) * k - p % TC_PLANES) * (TC_CORE / 16), idesc, k || p % TC_PLANES);
                tc_commit(b_free + 8 * buf);
                tc_commit(d_full + 8 * db);
            }
            tc_commit(drained);
            if (mbar_wait_bounded(drained, 0)) ok = false;
        }
    } else {                               // recombines: thread = output
        const PrimeConst pc = pcs[l];
        double c32 = 0, c64 = 0, c96 = 0;
        if (FP) {
            c32 = fp_reduce(4294967296.0, pc.qd, pc.qinvd);
            c64 = fp_modmul(c32, c32, pc.qd, pc.qinvd);
            c96 = fp_modmul(c64, c32, pc.qd, pc.qinvd);
        }
        const uint32_t row = tid & 127, half = warp >> 2, bp = mt * 128 + row;
        u64* out = acc + (size_t)bp * ctw + (size_t)l * N + c_first;
        for (uint32_t i0 = 0; i0 < coefs && ok; i0 += 4) {      // four coefficients make a full sector of every output row
            u64 r[4][4];
#pragma unroll
            for (uint32_t e = 0; e < 4; e++) {
                const uint32_t i = i0 + e, db = i & 1, du = i >> 1;
                if (ok && mbar_wait_bounded(d_full + 8 * db, du & 1)) ok = false;
                ok = __all_sync(0xFFFFFFFFu, ok);
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                uint32_t s[TC_ACCS][TC_GROUPS][4];       // group y of accumulator a: weight 256^(TC_PLANES a + y)
#pragma unroll
                for (int a = 0; a < TC_ACCS; a++)
#pragma unroll
                    for (int y = 0; y < TC_GROUPS; y++)
                        if (y < tc_groups(a)) tc_ld4(s[a][y], tmem + 256 * db + TC_ACC_COLS * a + 8 * y + 4 * half + ((32 * (warp & 3)) << 16));
                asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
                for (int a = 0; a < TC_ACCS; a++)
#pragma unroll
                    for (int y = 0; y < TC_GROUPS; y++)      // no use of a loaded word moves above the wait
                        if (y < tc_groups(a)) asm volatile("" : "+r"(s[a][y][0]), "+r"(s[a][y][1]), "+r"(s[a][y][2]), "+r"(s[a][y][3]));
                asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
                if (lane == 0) mbar_arrive(d_free + 8 * db);
#pragma unroll
                for (int n = 0; n < 4; n++) {
                    uint32_t v[13] = {};
#pragma unroll
                    for (int a = 0; a < TC_ACCS; a++)
#pragma unroll
                        for (int y = 0; y < TC_GROUPS; y++)
                            if (y < tc_groups(a)) v[TC_PLANES * a + y] += s[a][y][n];
                    r[n][e] = imma_reduce<FP>(v, pc, c32, c64, c96);
                }
            }
            if (ok && bp < bp_count) {
#pragma unroll
                for (uint32_t n = 0; n < 4; n++) {
                    const uint32_t tb = tbt * 4 + 2 * half + (n >> 1);
                    if (tb >= tbs) break;
                    u64* o = out + (size_t)tb * bp_count * ctw + (n & 1) * poly + i0;
                    // whole sectors: 16-byte stores took twice the time (59 against 35 ms with the arithmetic left out)
                    asm volatile("st.global.v4.b64 [%0], {%1, %2, %3, %4};" ::"l"(o), "l"(r[n][0]), "l"(r[n][1]), "l"(r[n][2]), "l"(r[n][3]) : "memory");
                }
            }
        }
    }
    if (!ok) atomicExch(status, 4u);
    __syncwarp();
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (warp == TC_OUT_WARPS) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 512;" ::"r"(tmem));
}

static uint32_t tc_buffers(uint32_t ksteps) {
    const uint32_t fit = (226u * 1024 - TC_A_BYTES(ksteps)) / TC_B_BYTES(ksteps);
    return fit < TC_BUFFERS ? fit : TC_BUFFERS;
}
// The left operand is worth its place in shared memory when at least 16 coefficients use it and half of a tile's 128 rows are filled; more than
// 192 terms do not fit.  8 token blocks x 189 terms at 6 limbs, here against packed.cu: 31 outputs 9.9 / 6.7 ms, 45 outputs 9.9 / 9.7, 64 outputs
// 10.0 / 12.7, 130 outputs (two tiles) 19.9 / 26.0, 210 outputs 20.1 / 40.8; one token block the same to a scale of 1/2.
bool bsgs_periodic_supported(uint32_t terms, uint32_t bp_count, uint32_t dshift) {
    return dshift >= 4 && (terms + 31) / 32 <= TC_MAX_KSTEPS && bp_count >= 64;
}
int bsgs_accumulate_periodic(fesc_ctx* ctx, const uint8_t* xpk, const uint8_t* dpk, u64* acc, uint32_t level, uint32_t tbs, uint32_t terms,
                             uint32_t bp_count, bool fp, uint32_t dshift, cudaStream_t st) {
    const uint32_t N = ctx->N, ksteps = (terms + 31) / 32, buffers = tc_buffers(ksteps);
    const dim3 grid((N >> dshift) * ((bp_count + 127) / 128) * ((tbs + 3) / 4), level);
    size_t smem = TC_A_BYTES(ksteps) + (size_t)buffers * TC_B_BYTES(ksteps);
    if (smem < 120 * 1024) smem = 120 * 1024;          // one CTA per SM: no CTA waits for another one's tensor memory
#define TC_LAUNCH(FP, KS)                                                                                                               \
    case KS: {                                                                                                                          \
        auto kern = k_bsgs_accumulate_periodic<FP, KS>;                                                                                 \
        FESC_CHECK_CUDA(ctx, cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));                       \
        kern<<<grid, TC_THREADS, smem, st>>>(xpk, dpk, acc, ctx->d_pc, N, level, tbs, bp_count, dshift, buffers, ctx->d_status);        \
    } break;
#define TC_PICK(FP) \
    switch (ksteps) { TC_LAUNCH(FP, 1) TC_LAUNCH(FP, 2) TC_LAUNCH(FP, 3) TC_LAUNCH(FP, 4) TC_LAUNCH(FP, 5) TC_LAUNCH(FP, 6) }
    prof_begin(ctx, PF_BSGS, st);
    if (fp) TC_PICK(true)
    else TC_PICK(false)
#undef TC_PICK
#undef TC_LAUNCH
    prof_end(ctx, PF_BSGS, st);
    FESC_CHECK_CUDA(ctx, cudaGetLastError());
    return FESC_OK;
}

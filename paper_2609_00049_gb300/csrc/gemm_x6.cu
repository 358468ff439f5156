// fp32 products on the 5th-generation tensor cores: C[M x N] = A[M x K]
// B[N x K]^T with both fp32 operands K-major and split into three bf16 planes,
//   a = a1 + a2 + a3  (8 significand bits each, rounded to nearest: exact),
//   a b ~= a1 b1 + (a1 b2 + a2 b1) + (a1 b3 + a2 b2 + a3 b1),
// six tcgen05.mma (kind::f16, bf16) per 16-wide K step.  The three dropped
// products are at most 2^-23 of |a b|, and bf16 has fp32's exponent range, so
// the operands need no scales.
//
// Accumulation: the tensor core rounds its fp32 accumulator towards zero, about
// one unit in the last place per MMA.  Each 32-wide K slice is therefore summed
// in TMEM on its own, the five small products first (their rounding is 2^-8 of
// the large one's) and then a1 b1, and the eight drain warps add the finished
// slice into fp32 registers (rounded to nearest) while the MMAs of the next
// slice fill the other of two TMEM accumulators.  An element then takes two
// truncations of a 32-term partial sum per slice, instead of K sequential
// roundings of the whole sum as an FFMA chain does: the error against fp64 is
// 0.2 to 0.45 of the CUDA-core product's at K = 8192 to 64.  The truncations
// all point towards zero, so what error remains would be a common factor of
// about 1 - 5e-8 on every output, which the window's difference of two passes
// does not average out as it does a random one (a window sweep's group scales
// moved by 2e-6 instead of 3e-7).  Three slices of every eight are therefore
// added with the factor 1 + 2^-23, which is the expected loss of dense random
// terms: with K a multiple of 256 their mean error is within 0.3e-8 of the
// output's scale.  It is not a bound for every operand: a product of one slice
// (K <= 32) keeps its -4.5e-8, one of two (K = 64) is left with +1.5e-8, a sum
// that one slice holds nearly all of (sparse or diagonal operands) takes that
// slice's -5e-8 or +1.2e-7, and sums of small integers, which the slices form
// exactly, are moved by up to one unit in the last place.
//
// One CTA owns a 128 x TN tile (TN = 256, or 128 where that fills the SMs
// better): warp 8 issues the TMA loads (one 3-D box per operand and stage: 32
// elements x rows x 3 planes, 64-byte rows, 64-byte swizzle), warp 9 the MMAs,
// warps 0-7 drain.  Per stage 12 MMAs of N = 256 take 1536 cycles, the drain of
// a 128 x 256 slice about 600, so the drain hides behind the MMAs.  Measured on
// 4096 x 3072, K = 1024: 108 us (240 TFLOP/s; six bf16 products per term bound it
// at 321) besides 14 us for the split, against 677 us on the fp32 CUDA cores.
#include "kernels.cuh"
#include "tc.cuh"

#include <mutex>

namespace realq {
namespace {

constexpr int TM = 128;
constexpr int KS = 32;                          // K elements per stage and per promoted slice
constexpr int NP = 3;                           // planes
constexpr int DRAIN_WARPS = 8;
constexpr int THREADS = (DRAIN_WARPS + 2) * 32;
constexpr int ROW_BYTES = KS * 2;               // 64-byte rows
constexpr int STG_PITCH = 33;
constexpr float kUp = 1.f + 1.1920929e-7f;      // 1 + 2^-23: see the bias of the truncations above

template <int TN>
struct X6Tile {
    static constexpr int STAGES = TN == 256 ? 3 : 4;
    static constexpr int PLANE_A = TM * ROW_BYTES;
    static constexpr int PLANE_B = TN * ROW_BYTES;
    static constexpr int STAGE_BYTES = NP * (PLANE_A + PLANE_B);
    static constexpr int SMEM = STAGES * STAGE_BYTES + 1024 + 256;
    static constexpr uint32_t IDESC = tc::idesc_bf16_f32(TM, TN, 0, 0);
    static_assert(SMEM <= 232448, "shared memory of the bf16x6 product");
    static_assert(STAGES * STAGE_BYTES >= DRAIN_WARPS * 32 * STG_PITCH * 4, "epilogue staging fits the ring");
};

template <int TN>
__global__ void __launch_bounds__(THREADS, 1)
    gemm_x6_kernel(const __grid_constant__ CUtensorMap ma, const __grid_constant__ CUtensorMap mb, int64_t M, int64_t N,
                   int64_t K, int b_row0, const X6Epi e, int *err) {
    using TL = X6Tile<TN>;
    constexpr int STAGES = TL::STAGES;
    extern __shared__ uint8_t smem_raw[];
    uint8_t *smem = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    uint64_t *full = reinterpret_cast<uint64_t *>(smem + STAGES * TL::STAGE_BYTES);
    uint64_t *empty = full + STAGES;
    uint64_t *accf = empty + STAGES;            // [2] accumulator b holds a finished slice
    uint64_t *acce = accf + 2;                  // [2] accumulator b has been drained
    uint64_t *drain = acce + 2;                 // the MMA thread's last commit
    uint32_t *tslot = reinterpret_cast<uint32_t *>(drain + 1);
    volatile int *abort_flag = reinterpret_cast<volatile int *>(tslot + 1);

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    // tiles in groups of 8 row tiles, as the x3 products: the CTAs resident
    // together share their operand rows through L2
    int64_t i0, j0;
    {
        const int64_t nx = gridDim.x, ny = gridDim.y, pid = (int64_t)blockIdx.y * nx + blockIdx.x;
        constexpr int64_t GROUP = 8;
        const int64_t per = GROUP * nx, first = (pid / per) * GROUP;
        const int64_t gm = (ny - first) < GROUP ? (ny - first) : GROUP;
        i0 = (first + (pid % per) % gm) * TM;
        j0 = ((pid % per) / gm) * TN;
    }
    if (e.mode == X6_UPPER && e.joff + j0 + TN <= i0) return;   // wholly below the diagonal (uniform over the CTA)
    // triangular operands shorten the K range: a_lo A(i, k) = 0 for k < i,
    // b_lo B(j, k) = 0 for k < j (32 bits hold it: the operands' k is checked)
    int kbeg = 0;
    if (e.a_lo && i0 > kbeg) kbeg = (int)i0;
    if (e.b_lo && j0 > kbeg) kbeg = (int)j0;
    kbeg = kbeg / KS * KS;
    const int nk = K > kbeg ? (int)((K - kbeg + KS - 1) / KS) : 0;

    if (threadIdx.x == 0) {
        for (int s = 0; s < STAGES; ++s) {
            tc::mbar_init(tc::smem_u32(&full[s]), 1);
            tc::mbar_init(tc::smem_u32(&empty[s]), 1);
        }
        for (int b = 0; b < 2; ++b) {
            tc::mbar_init(tc::smem_u32(&accf[b]), 1);
            tc::mbar_init(tc::smem_u32(&acce[b]), DRAIN_WARPS);
        }
        tc::mbar_init(tc::smem_u32(drain), 1);
        *abort_flag = 0;
        tc::fence_barrier_init();
        tc::prefetch_tmap(&ma);
        tc::prefetch_tmap(&mb);
    }
    if (warp == 0) tc::tmem_alloc(tc::smem_u32(tslot), 2 * TN);
    tc::fence_before_sync();
    __syncthreads();
    tc::fence_after_sync();
    const uint32_t tmem = *tslot;

    float acc[TN / 2];
#pragma unroll
    for (int c = 0; c < TN / 2; ++c) acc[c] = 0.f;
    bool good = true;

    if (warp == DRAIN_WARPS) {
        if (lane == 0) {
            // ---------------- TMA producer ----------------
            int it = 0;
            for (; it < nk; ++it) {
                const int s = it % STAGES;
                const uint32_t r = (uint32_t)(it / STAGES);
                if (!tc::mbar_wait(tc::smem_u32(&empty[s]), (r & 1u) ^ 1u, abort_flag)) {
                    *abort_flag = 1;
                    break;
                }
                const uint32_t fb = tc::smem_u32(&full[s]);
                tc::mbar_arrive_expect_tx(fb, TL::STAGE_BYTES);
                const int x = kbeg + it * KS;
                const uint32_t base = tc::smem_u32(smem + s * TL::STAGE_BYTES);
                tc::tma_load_3d(base, &ma, fb, x, (int)i0, 0);
                tc::tma_load_3d(base + NP * TL::PLANE_A, &mb, fb, x, b_row0 + (int)j0, 0);
            }
            if (*abort_flag) {
                int never = 0;
                for (int k = (it > STAGES ? it - STAGES : 0); k < it; ++k)
                    tc::mbar_wait(tc::smem_u32(&full[k % STAGES]), (uint32_t)(k / STAGES) & 1u, &never, 100000000ull);
            }
        }
    } else if (warp == DRAIN_WARPS + 1) {
        if (lane == 0 && nk > 0) {
            // ---------------- MMA issuer ----------------
            for (int it = 0; it < nk; ++it) {
                const int s = it % STAGES, b = it & 1;
                const uint32_t r = (uint32_t)(it / STAGES);
                if (it >= 2 && !tc::mbar_wait(tc::smem_u32(&acce[b]), (uint32_t)((it >> 1) - 1) & 1u, abort_flag)) {
                    *abort_flag = 1;
                    break;
                }
                if (!tc::mbar_wait(tc::smem_u32(&full[s]), r & 1u, abort_flag)) {
                    *abort_flag = 1;
                    break;
                }
                tc::fence_after_sync();
                const uint32_t d = tmem + (uint32_t)(b * TN);
                const uint32_t ab = tc::smem_u32(smem + s * TL::STAGE_BYTES), bb = ab + NP * TL::PLANE_A;
                auto da = [&](int p, int k) { return tc::smem_desc(ab + p * TL::PLANE_A + k * 32, 16, 512, tc::SW_64B); };
                auto db = [&](int p, int k) { return tc::smem_desc(bb + p * TL::PLANE_B + k * 32, 16, 512, tc::SW_64B); };
                // the small products of both K steps first, the large ones last
#pragma unroll
                for (int k = 0; k < KS / 16; ++k) {
                    tc::mma_bf16_ss(d, da(2, k), db(0, k), TL::IDESC, k > 0 ? 1u : 0u);
                    tc::mma_bf16_ss(d, da(1, k), db(1, k), TL::IDESC, 1u);
                    tc::mma_bf16_ss(d, da(0, k), db(2, k), TL::IDESC, 1u);
                }
#pragma unroll
                for (int k = 0; k < KS / 16; ++k) {
                    tc::mma_bf16_ss(d, da(1, k), db(0, k), TL::IDESC, 1u);
                    tc::mma_bf16_ss(d, da(0, k), db(1, k), TL::IDESC, 1u);
                }
#pragma unroll
                for (int k = 0; k < KS / 16; ++k) tc::mma_bf16_ss(d, da(0, k), db(0, k), TL::IDESC, 1u);
                tc::mma_commit(tc::smem_u32(&empty[s]));
                tc::mma_commit(tc::smem_u32(&accf[b]));
            }
            // every MMA issued has retired before TMEM is freed
            tc::mma_commit(tc::smem_u32(drain));
            int never = 0;
            tc::mbar_wait(tc::smem_u32(drain), 0u, &never, 100000000ull);
        }
    } else {
        // ------- drain warps: TMEM slice -> fp32 registers (lane quarter, column half) -------
        const uint32_t lane_base = (uint32_t)((warp & 3) * 32) << 16;
        const uint32_t col_base = (uint32_t)((warp >> 2) * (TN / 2));
        if (e.mode != X6_STORE || e.R) {
            // the tile that the epilogue combines with, into L2 while the MMAs
            // run: one 128-byte line per thread and step
            const float *src = e.mode == X6_STORE ? e.R : e.C;
            const int64_t lds = e.mode == X6_STORE ? e.ldr : e.ldc;
            const int64_t jm = N < j0 + TN ? N : j0 + TN;
            for (int l = threadIdx.x; l < TM * (TN / 32); l += DRAIN_WARPS * 32) {
                const int64_t gi = i0 + l / (TN / 32), gj = j0 + (l % (TN / 32)) * 32;
                if (gi < M && gj < jm) asm volatile("prefetch.global.L2 [%0];" ::"l"(src + gi * lds + gj));
            }
        }
        for (int it = 0; it < nk; ++it) {
            const int b = it & 1;
            const bool ok = tc::mbar_wait(tc::smem_u32(&accf[b]), (uint32_t)(it >> 1) & 1u, abort_flag);
            if (!__all_sync(0xffffffffu, ok)) {
                good = false;
                break;
            }
            tc::fence_after_sync();
            const float up = ((0x52 >> (it & 7)) & 1) ? kUp : 1.f;   // slices 1, 4 and 6 of eight
#pragma unroll
            for (int c0 = 0; c0 < TN / 2; c0 += 16) {
                uint32_t v[16];
                tc::tmem_ld_32x32b_x16(tmem + lane_base + (uint32_t)(b * TN) + col_base + (uint32_t)c0, v);
#pragma unroll
                for (int q = 0; q < 16; ++q) acc[c0 + q] = fmaf(__uint_as_float(v[q]), up, acc[c0 + q]);
            }
            tc::fence_before_sync();
            __syncwarp();
            if (lane == 0) tc::mbar_arrive(tc::smem_u32(&acce[b]));
        }
    }
    __syncwarp();
    const bool all_good = __syncthreads_and(good && !*abort_flag) != 0;
    if (!all_good && threadIdx.x == 0) *abort_flag = 1;
    // ---------------- epilogue: registers -> shared memory -> global ----------------
    // (the ring is free: every stage loaded has been multiplied; each warp
    // stages 32 x 32 blocks so that the rows of C are accessed coalesced)
    if (warp < DRAIN_WARPS && all_good) {
        float *st = reinterpret_cast<float *>(smem) + warp * 32 * STG_PITCH;
        const int64_t gi0 = i0 + (warp & 3) * 32;
#pragma unroll
        for (int c0 = 0; c0 < TN / 2; c0 += 32) {
            const int64_t gj = j0 + (warp >> 2) * (TN / 2) + c0 + lane;
            // rows 0 .. top - 1 of the block are written; what C is combined
            // with is read first, 16 rows at a time (a load after a store to C
            // would wait for it)
            const int rows = (int)(M - gi0 < 32 ? (M - gi0 > 0 ? M - gi0 : 0) : 32);
            const bool upper = e.mode == X6_UPPER;
            const bool fold = upper || (e.mode == X6_ADD && gj >= e.nstore) || (e.mode == X6_STORE && e.R);
            const float *src = (e.mode == X6_STORE ? e.R : e.C) + gi0 * (e.mode == X6_STORE ? e.ldr : e.ldc) + gj;
            const int64_t lds = e.mode == X6_STORE ? e.ldr : e.ldc;
            int top = upper && gj + e.joff - gi0 + 1 < rows ? (int)(gj + e.joff - gi0 + 1) : rows;
            if (gj >= N) top = 0;
#pragma unroll
            for (int q = 0; q < 32; ++q) st[lane * STG_PITCH + q] = acc[c0 + q];
            __syncwarp();
            float *dst = e.C + gi0 * e.ldc + gj;
#pragma unroll 1
            for (int r0 = 0; r0 < top; r0 += 16) {
                float old[16];
#pragma unroll
                for (int u = 0; u < 16; ++u) old[u] = fold && r0 + u < top ? src[u * lds] : 0.f;
#pragma unroll
                for (int u = 0; u < 16; ++u)
                    if (r0 + u < top) dst[u * e.ldc] = old[u] + e.alpha * st[(r0 + u) * STG_PITCH + lane];
                src += 16 * lds;
                dst += 16 * e.ldc;
            }
            __syncwarp();
        }
    }
    if (!all_good && threadIdx.x == 0 && err) atomicOr(err, ST_TIMEOUT);
    tc::fence_before_sync();
    __syncthreads();
    if (warp == 0) tc::tmem_dealloc(tmem, 2 * TN);
}

// The three bf16 parts of v, rounded to nearest (a finite value whose first
// part would round to infinity is truncated instead; the parts of a
// non-finite value are the value and zeros, so that a product with an infinite
// operand is not finite: infinite where the other's three parts have one sign
// and none is zero, else NaN, where the fp32 product gives infinity).
__device__ __forceinline__ void split3(float v, __nv_bfloat16 &a, __nv_bfloat16 &b, __nv_bfloat16 &c) {
    a = __float2bfloat16_rn(v);
    float h = __bfloat162float(a);
    if (isinf(h) && !isinf(v)) {
        h = __uint_as_float(__float_as_uint(v) & 0xFFFF0000u);
        a = __float2bfloat16_rn(h);
    }
    const float r = isfinite(v) ? v - h : 0.f;
    b = __float2bfloat16_rn(r);
    c = __float2bfloat16_rn(r - __bfloat162float(b));
}

// One operand to split: src (rows x cols, row stride lds) into planes of its
// rows (dst[r * ldd + c]), or of its columns (trans: dst[c * ldd + r]).
// CTA t of a job takes a 32 x 32 tile, or 1024 elements of the rows form.
struct SplitJob {
    const float *src;
    __nv_bfloat16 *dst;
    int64_t lds, rows, cols, ldd, plane, tiles, tiles_c;
    int trans;
};

__global__ void __launch_bounds__(256) split3_kernel(const SplitJob ja, const SplitJob jb) {
    const bool second = (int64_t)blockIdx.x >= ja.tiles;
    const SplitJob &j = second ? jb : ja;
    const int64_t t = (int64_t)blockIdx.x - (second ? ja.tiles : 0);
    if (!j.trans) {
        const int64_t c4 = (j.cols + 3) / 4;
        const int64_t idx = t * 256 + threadIdx.x;
        if (idx >= j.rows * c4) return;
        const int64_t r = idx / c4, c = (idx % c4) * 4;
        const float *s = j.src + r * j.lds + c;
        float v[4];
        if (c + 3 < j.cols && ((reinterpret_cast<uintptr_t>(s) & 15) == 0)) {
            const float4 q = *reinterpret_cast<const float4 *>(s);
            v[0] = q.x; v[1] = q.y; v[2] = q.z; v[3] = q.w;
        } else {
#pragma unroll
            for (int u = 0; u < 4; ++u) v[u] = c + u < j.cols ? s[u] : 0.f;
        }
        __nv_bfloat162 p[NP][2];
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            split3(v[2 * u], p[0][u].x, p[1][u].x, p[2][u].x);
            split3(v[2 * u + 1], p[0][u].y, p[1][u].y, p[2][u].y);
        }
        // (ldd is a multiple of 8, so it covers the columns rounded up to 4)
#pragma unroll
        for (int k = 0; k < NP; ++k)
            *reinterpret_cast<uint2 *>(j.dst + k * j.plane + r * j.ldd + c) = *reinterpret_cast<const uint2 *>(p[k]);
        return;
    }
    __shared__ float tile[32][33];
    const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
    const int64_t tr = t / j.tiles_c, tcol = t % j.tiles_c;
    const int64_t c = tcol * 32 + tx;
#pragma unroll
    for (int q = 0; q < 32; q += 8) {
        const int64_t r = tr * 32 + ty + q;
        tile[ty + q][tx] = (r < j.rows && c < j.cols) ? j.src[r * j.lds + c] : 0.f;
    }
    __syncthreads();
    // each thread writes two consecutive rows of one column of src
    const int rr = (threadIdx.x & 15) * 2, cy = threadIdx.x >> 4;
#pragma unroll
    for (int q = 0; q < 32; q += 16) {
        const int64_t cc = tcol * 32 + cy + q, r = tr * 32 + rr;
        if (cc >= j.cols || r >= j.rows) continue;
        __nv_bfloat162 p[NP];
        split3(tile[rr][cy + q], p[0].x, p[1].x, p[2].x);
        split3(tile[rr + 1][cy + q], p[0].y, p[1].y, p[2].y);
        // (ldd is a multiple of 8, so it covers the rows rounded up to 2)
#pragma unroll
        for (int k = 0; k < NP; ++k)
            *reinterpret_cast<__nv_bfloat162 *>(j.dst + k * j.plane + cc * j.ldd + r) = p[k];
    }
}

SplitJob job_of(const X6Split &x) {
    SplitJob j{x.src, x.dst, x.lds, x.rows, x.cols, x.ldd, x.plane, 0, ceil_div(x.cols, 32), x.trans};
    if (x.rows > 0 && x.cols > 0)
        j.tiles = x.trans ? (int64_t)ceil_div(x.rows, 32) * j.tiles_c : ceil_div(x.rows * ((x.cols + 3) / 4), 256);
    return j;
}

realq_status_t check_planes(const X6Planes &p, const char *name) {
    if (p.ld % 8 != 0 || p.plane % 8 != 0 || (reinterpret_cast<uintptr_t>(p.p) & 15) || p.rows <= 0 || p.k <= 0 ||
        p.rows >= (1ll << 31) || p.k >= (1ll << 31))
        return fail(REALQ_ERR_INVALID_ARG, "%s: bf16 planes need 16-byte rows and bases", name);
    return REALQ_OK;
}

template <int TN>
realq_status_t launch_x6(cudaStream_t s, const X6Planes &A, const X6Planes &B, int64_t M, int64_t N, int64_t K,
                         int b_row0, const X6Epi &e, int *err) {
    CUtensorMap ma, mb;
    CUresult r = encode_tmap_3d_bf16(&ma, A.p, (uint64_t)A.k, (uint64_t)A.rows, NP, (uint64_t)A.ld * 2,
                                     (uint64_t)A.plane * 2, KS, TM, NP);
    if (r == CUDA_SUCCESS)
        r = encode_tmap_3d_bf16(&mb, B.p, (uint64_t)B.k, (uint64_t)B.rows, NP, (uint64_t)B.ld * 2,
                                (uint64_t)B.plane * 2, KS, TN, NP);
    if (r != CUDA_SUCCESS) return fail(REALQ_ERR_CUDA, "cuTensorMapEncodeTiled (bf16 planes) failed (%d)", (int)r);
    REALQ_TRY(set_smem_limit(reinterpret_cast<const void *>(gemm_x6_kernel<TN>), X6Tile<TN>::SMEM));
    const dim3 grid((unsigned)ceil_div(N, TN), (unsigned)ceil_div(M, TM));
    gemm_x6_kernel<TN><<<grid, THREADS, X6Tile<TN>::SMEM, s>>>(ma, mb, M, N, K, b_row0, e, err);
    return REALQ_OK;
}

}  // namespace

realq_status_t split3(cudaStream_t s, const X6Split &a, const X6Split *b) {
    const SplitJob ja = job_of(a), jb = b ? job_of(*b) : SplitJob{};
    for (const SplitJob *j : {&ja, &jb})
        if (j->tiles > 0 && (j->ldd % 8 != 0 || j->plane % 8 != 0 || (reinterpret_cast<uintptr_t>(j->dst) & 15)))
            return fail(REALQ_ERR_INVALID_ARG, "bf16 split: planes need 16-byte rows and bases");
    if (ja.tiles + jb.tiles <= 0) return REALQ_OK;
    if (ja.tiles + jb.tiles > 0x7FFFFFFFll) return fail(REALQ_ERR_UNSUPPORTED, "bf16 split: operand too large");
    {
        Launch L("bf16_split", s);
        split3_kernel<<<(unsigned)(ja.tiles + jb.tiles), 256, 0, s>>>(ja, jb);
    }
    return check_launch("bf16_split");
}

realq_status_t gemm_x6(cudaStream_t s, const X6Planes &A, const X6Planes &B, int64_t M, int64_t N, int64_t K,
                       int64_t b_row0, const X6Epi &e, int *err, const char *name) {
    if (M <= 0 || N <= 0) return REALQ_OK;
    REALQ_TRY(check_planes(A, name));
    REALQ_TRY(check_planes(B, name));
    // the 128 x 256 tile where it leaves no more of the last wave idle than it
    // saves in operand traffic (a 128 x 128 tile takes about 0.6 of its time)
    const int sms = num_sms();
    const int64_t rows = ceil_div(M, TM);
    const int64_t w256 = ceil_div(rows * ceil_div(N, 256), sms), w128 = ceil_div(rows * ceil_div(N, 128), sms);
    {
        Launch L(name, s);
        if (10 * w256 <= 6 * w128)
            REALQ_TRY(launch_x6<256>(s, A, B, M, N, K, (int)b_row0, e, err));
        else
            REALQ_TRY(launch_x6<128>(s, A, B, M, N, K, (int)b_row0, e, err));
    }
    return check_launch(name);
}

}  // namespace realq

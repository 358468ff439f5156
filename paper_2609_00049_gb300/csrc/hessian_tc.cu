// Step a2 (Sec. 3.2) on the 5th-generation tensor cores: H_sum += X̂^T X̂ for
// bf16 calibration activations.
//
// A pair of CTAs (a cluster of two, cta_group::2) owns one 256 x 256 tile (256
// channels i by 256 channels j, on or below the diagonal) of H and a contiguous
// range of tokens; each CTA loads its 128 channels of A and its 128 channels of
// B, the leader issues tcgen05.mma of M = 256, N = 256, K = 16 for both, and each
// CTA's TMEM takes its own 128 rows.  X̂ is token-major (T x n), so both MMA
// operands are read MN-major straight from the activation rows: a TMA box of 64
// tokens x 64 channels (128-byte rows, 128-byte swizzle) is one canonical
// MN-major atom stack; two boxes make a CTA's 128 channels of an operand (LBO =
// 8 KB between boxes, SBO = 1 KB between 8-token groups).
//
// What bounds it: a 128 x 256 tile per CTA reads 12 KB of shared memory per MMA
// of 128 cycles and is written 48 KB per four of them, 192 bytes per cycle
// against the 128 that an SM serves, so it topped out at two thirds of the
// tensor pipe.  The pair halves B's share: 64 + 64 bytes per cycle.
//
// Precision: the tensor core's fp32 accumulation loses about one unit in the
// last place per accumulated MMA, in one direction, so a TMEM accumulator that
// takes all 2^18 tokens of a calibration set (2^14 MMAs) drifts by ~1e-3 of
// the entry.  The accumulation is therefore promoted: TMEM holds two 128 x 256
// accumulators (per CTA), the MMA issuer switches between them every 640 tokens
// (CHUNK_STAGES), and the eight drain warps add each finished chunk into fp32
// registers (IEEE adds) while the other accumulator fills.
//
// Roles (320 threads per CTA): warp 8 lane 0 issues the CTA's TMA loads into a
// STAGES-deep ring (counted on the leader's barriers), warp 9 lane 0 of the
// leader issues the MMAs and frees the stages of both CTAs with
// tcgen05.commit; warps 0-7 drain the CTA's accumulators (warp w owns TMEM
// lanes 32 (w % 4).. and columns 128 (w / 4)..) and finally add their piece to H
// (mirrored below the diagonal block), or store it as a partial sum when tokens
// are split; either way through a shared-memory block, so that a row's accesses
// coalesce (one row per thread cost 40 us at n = 1024).
//
// A width that is no multiple of 256 leaves a last block of n % 256 channels.
// Its tiles take it as the columns (the MMA's N, down to 32), also where it
// belongs on the rows: such a tile is computed transposed ("swap") and stored
// so.  At n = 2056 the last block's tiles are 26 of 126 and cost 0.3 of a full
// one each.
//
// The cross tiles compute the full (non-symmetric) product X_Cᵀ X_B: the cross
// moment of the perturbed-input surrogate is D = X̂ᵀX̂ - XᵀX̂.  With token splits
// both products run in one launch over the same splits and the reduction
// subtracts their sums (kept in two floats each) before it adds to D, so that
// little of D is lost to the size of its two parts; without splits, or where the
// workspace holds one product's partial sums only, the symmetric sum is also
// added to D and a second launch subtracts.
// Every wait is bounded; on a timeout in either CTA of a pair the whole tile is
// written as NaN (so the factorisation of H reports a non-finite pivot), the
// workspace status word gets ST_TIMEOUT, and the kernel still frees TMEM and
// returns.
#include "kernels.cuh"
#include "tc.cuh"

#include <algorithm>
#include <cmath>
#include <mutex>
#include <type_traits>

namespace realq {
namespace {

constexpr int TM = 128;                          // tile rows of one CTA (channels i)
constexpr int TN = 256;                          // tile rows of the pair, and tile columns (channels j)
constexpr int KSTAGE = 64;                       // tokens per pipeline stage
constexpr int STAGES = 6;
// 640 tokens per TMEM accumulator pass, with and without D: H then has the same
// bits whether or not D is asked for.  D, the small difference of two large
// sums, magnifies the accumulator's rounding and sets the length: it is the
// longest with which D's error against 64 bits (2-norm, mean over 6 to 14 seeds) is
// no larger at any measured shape than with one CTA per tile and 1024 tokens.
// n = 2056, T = 50,001: 8.5e-6 so; here 512 tokens 6.3e-6, 640 7.3e-6, 704 8.9e-6,
// 1024 8.7e-6.  n = 1024, T = 65,536: 8.3e-6; 4.2e-6, 5.1e-6, 6.6e-6, 7.3e-6.
constexpr int CHUNK_STAGES = 10;
constexpr int DRAIN_WARPS = 8;                   // two per TMEM lane quarter, 128 columns each
constexpr int THREADS = (DRAIN_WARPS + 2) * 32;  // + the TMA warp and the MMA warp
constexpr int BOX_BYTES = 64 * KSTAGE * 2;       // one TMA box (64 channels x 64 tokens)
constexpr int A_BYTES = TM * KSTAGE * 2;         // 2 boxes
constexpr int B_BYTES = TM * KSTAGE * 2;         // 2 boxes: this CTA's half of the columns
constexpr int STAGE_BYTES = A_BYTES + B_BYTES;
constexpr int SMEM_BYTES = STAGES * STAGE_BYTES + 1024 + 256;
constexpr unsigned FULL = 0xFFFFFFFFu;

// The lower tiles (ti >= tj of nt x nt) in groups of 4 tile rows: a group's tiles
// column by column (within a column, its rows that reach it), so that the CTAs
// resident at one time cover a compact block of the product and share their
// channel blocks through L2.  A bijection onto {(ti, tj): tj <= ti < nt}.
__device__ __forceinline__ void lower_tile(int64_t idx, int nt, int &ti, int &tj) {
    constexpr int G = 4;
    int r0 = 0;
    for (;; r0 += G) {
        const int r1 = min(r0 + G, nt);
        const int64_t c = (int64_t)r1 * (r1 + 1) / 2 - (int64_t)r0 * (r0 + 1) / 2;
        if (idx < c || r1 >= nt) break;
        idx -= c;
    }
    const int r1 = min(r0 + G, nt);
    for (int j = 0;; ++j) {
        const int lo = max(r0, j);
        const int cnt = r1 > lo ? r1 - lo : 0;
        if (cnt == 0) {   // (not reached for idx < nt (nt + 1) / 2)
            ti = r1 - 1;
            tj = 0;
            return;
        }
        if (idx < cnt) {
            ti = lo + (int)idx;
            tj = j;
            return;
        }
        idx -= cnt;
    }
}

// A tile of the launch: A's 256-channel block ti, B's block tj with ncol (32 ..
// 256) columns; cross or symmetric; swap: stored transposed.
struct HessTile {
    int ti, tj, ncol;
    bool cross, swap;
};
struct HessGrid {
    int64_t n;
    int nf, rem;           // full 256-channel blocks, channels of the last one
    int64_t nsym, ncross;  // tiles
};
inline HessGrid hess_grid(int64_t n, bool sym, bool cross) {
    HessGrid g{n, (int)(n / TN), (int)(n % TN), 0, 0};
    const int64_t r = g.rem ? 1 : 0, nf = g.nf;
    if (sym) g.nsym = nf * (nf + 1) / 2 + r * (nf + 1);
    if (cross) g.ncross = nf * nf + r * (2 * nf + 1);
    return g;
}
__device__ __forceinline__ HessTile hess_tile(const HessGrid &g, int64_t idx) {
    HessTile t{0, 0, TN, false, false};
    const int nlast = (g.rem + 31) / 32 * 32;
    if (idx < g.nsym) {
        const int64_t full = (int64_t)g.nf * (g.nf + 1) / 2;
        if (idx < full) {
            lower_tile(idx, g.nf, t.ti, t.tj);
        } else {
            t.ti = (int)(idx - full);
            t.tj = g.nf;
            t.ncol = nlast;
            t.swap = t.ti < g.nf;
        }
        return t;
    }
    idx -= g.nsym;
    t.cross = true;
    const int64_t full = (int64_t)g.nf * g.nf;
    if (idx < full) {
        // groups of 4 tile rows, column by column
        constexpr int G = 4;
        const int64_t per = (int64_t)G * g.nf;
        const int r0 = (int)(idx / per) * G, gm = min(G, g.nf - r0);
        t.ti = r0 + (int)(idx % per) % gm;
        t.tj = (int)((idx % per) / gm);
        return t;
    }
    idx -= full;
    t.tj = g.nf;
    t.ncol = nlast;
    t.swap = idx > g.nf;                                     // (the last row block's other tiles)
    t.ti = (int)(t.swap ? idx - g.nf - 1 : idx);
    return t;
}

__global__ void __launch_bounds__(THREADS, 1)
    hess_tc_kernel(const __grid_constant__ CUtensorMap mapA, const __grid_constant__ CUtensorMap mapB,
                   const __grid_constant__ CUtensorMap mapC, const HessGrid grid, int64_t T, int64_t tper, float *H,
                   float *H2, float *part, float *partC, float sign, int chunk_stages, int *err) {
    extern __shared__ uint8_t smem_raw[];
    uint8_t *smem = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    uint64_t *full = reinterpret_cast<uint64_t *>(smem + STAGES * STAGE_BYTES);
    uint64_t *empty = full + STAGES;
    uint64_t *accf = empty + STAGES;             // [2] accumulator b holds a finished chunk
    uint64_t *acce = accf + 2;                   // [2] accumulator b has been drained
    uint64_t *drain = acce + 2;                  // the MMA thread's last commit
    uint32_t *tslot = reinterpret_cast<uint32_t *>(drain + 1);
    volatile int *abort_flag = reinterpret_cast<volatile int *>(tslot + 1);

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int64_t n = grid.n;
    const uint32_t rank = tc::cluster_rank();
    const bool leader = rank == 0;
    const HessTile tl = hess_tile(grid, blockIdx.x / 2);
    // this CTA's 128 rows of the tile, and its half of the columns as an operand
    const int i0 = tl.ti * TN + (int)rank * TM, jl = tl.tj * TN + (int)rank * (tl.ncol / 2);
    const int bboxes = (tl.ncol / 2 + 63) / 64;
    const int64_t t_begin = (int64_t)blockIdx.y * tper;
    const int64_t t_end = min(T, t_begin + tper);
    const int nk = t_end > t_begin ? (int)((t_end - t_begin + KSTAGE - 1) / KSTAGE) : 0;
    const int nch = (nk + chunk_stages - 1) / chunk_stages;

    if (threadIdx.x == 0) {
        for (int s = 0; s < STAGES; ++s) {
            tc::mbar_init(tc::smem_u32(&full[s]), 1);
            tc::mbar_init(tc::smem_u32(&empty[s]), 1);
        }
        for (int b = 0; b < 2; ++b) {
            tc::mbar_init(tc::smem_u32(&accf[b]), 1);
            tc::mbar_init(tc::smem_u32(&acce[b]), 2 * DRAIN_WARPS);   // both CTAs' (the leader's is waited on)
        }
        tc::mbar_init(tc::smem_u32(drain), 1);
        *abort_flag = 0;
        tc::fence_barrier_init();
        tc::prefetch_tmap(&mapA);
        tc::prefetch_tmap(&mapB);
        tc::prefetch_tmap(&mapC);
    }
    if (warp == 0) tc::tmem_alloc_pair(tc::smem_u32(tslot), 2 * TN);
    tc::fence_before_sync();
    __syncthreads();
    tc::cluster_sync();   // the peer's barriers are initialized
    tc::fence_after_sync();
    const uint32_t tmem = *tslot;

    float acc[128];
#pragma unroll
    for (int c = 0; c < 128; ++c) acc[c] = 0.f;
    bool good = true;

    if (warp == DRAIN_WARPS) {
        if (lane == 0) {
            // ---------------- TMA producer ----------------
            // symmetric: A from mapA, B from mapB; cross: A from mapC, B from
            // mapB, the other way round when the tile is stored transposed
            const CUtensorMap *ma = !tl.cross ? &mapA : (tl.swap ? &mapB : &mapC);
            const CUtensorMap *mb = tl.cross && tl.swap ? &mapC : &mapB;
            for (int it = 0; it < nk; ++it) {
                const int s = it % STAGES;
                const uint32_t r = (uint32_t)(it / STAGES);
                if (!tc::mbar_wait(tc::smem_u32(&empty[s]), (r & 1u) ^ 1u, abort_flag)) {
                    *abort_flag = 1;
                    break;
                }
                // (both CTAs' bytes are counted on the leader's barrier)
                const uint32_t fb = tc::mapa(tc::smem_u32(&full[s]), 0);
                if (leader) tc::mbar_arrive_expect_tx(tc::smem_u32(&full[s]), 2 * (A_BYTES + bboxes * BOX_BYTES));
                const int y = (int)(t_begin + (int64_t)it * KSTAGE);
                const uint32_t a = tc::smem_u32(smem + s * STAGE_BYTES);
                tc::tma_load_2d_pair(a, ma, fb, i0, y);
                tc::tma_load_2d_pair(a + BOX_BYTES, ma, fb, i0 + 64, y);
                for (int q = 0; q < bboxes; ++q) tc::tma_load_2d_pair(a + A_BYTES + q * BOX_BYTES, mb, fb, jl + 64 * q, y);
            }
        }
    } else if (warp == DRAIN_WARPS + 1) {
        if (lane == 0 && leader) {
            // ---------------- MMA issuer ----------------
            const uint32_t idesc = tc::idesc_bf16_f32(2 * TM, (uint32_t)tl.ncol, 1, 1);
            for (int c = 0; c < nch && !*abort_flag; ++c) {
                const int b = c & 1;
                if (c >= 2 && !tc::mbar_wait(tc::smem_u32(&acce[b]), (uint32_t)((c >> 1) - 1) & 1u, abort_flag)) {
                    *abort_flag = 1;
                    break;
                }
                tc::fence_after_sync();
                const uint32_t d = tmem + (uint32_t)(b * TN);
                const int it_end = min(nk, (c + 1) * chunk_stages);
                for (int it = c * chunk_stages; it < it_end; ++it) {
                    const int s = it % STAGES;
                    const uint32_t r = (uint32_t)(it / STAGES);
                    if (!tc::mbar_wait(tc::smem_u32(&full[s]), r & 1u, abort_flag)) {
                        *abort_flag = 1;
                        break;
                    }
                    tc::fence_after_sync();
                    const uint32_t a = tc::smem_u32(smem + s * STAGE_BYTES);
                    const uint32_t bop = a + A_BYTES;
                    const bool first = it == c * chunk_stages;
#pragma unroll
                    for (int k = 0; k < KSTAGE / 16; ++k) {
                        const uint64_t da = tc::smem_desc(a + k * 2048, BOX_BYTES, 1024, tc::SW_128B);
                        const uint64_t db = tc::smem_desc(bop + k * 2048, BOX_BYTES, 1024, tc::SW_128B);
                        tc::mma_f16_pair(d, da, db, idesc, (first && k == 0) ? 0u : 1u);
                    }
                    tc::mma_commit_pair(tc::smem_u32(&empty[s]));
                }
                // (a chunk cut short is not announced)
                if (!*abort_flag) tc::mma_commit_pair(tc::smem_u32(&accf[b]));
            }
            // every MMA issued has retired before TMEM is freed
            tc::mma_commit_pair(tc::smem_u32(drain));
            int never = 0;
            tc::mbar_wait(tc::smem_u32(drain), 0u, &never, 100000000ull);
        }
    } else {
        // ------- drain warps: TMEM chunk -> fp32 registers (lane quarter, column half) -------
        const uint32_t lane_base = (uint32_t)((warp & 3) * 32) << 16;
        const int col_base = (warp >> 2) * 128;
        for (int c = 0; c < nch; ++c) {
            const int b = c & 1;
            const bool ok = tc::mbar_wait(tc::smem_u32(&accf[b]), (uint32_t)(c >> 1) & 1u, abort_flag);
            if (!__all_sync(FULL, ok)) {
                good = false;
                break;
            }
            tc::fence_after_sync();
#pragma unroll
            for (int c0 = 0; c0 < 128; c0 += 16) {
                if (col_base + c0 < tl.ncol) {
                    uint32_t v[16];
                    tc::tmem_ld_32x32b_x16(tmem + lane_base + (uint32_t)(b * TN + col_base + c0), v);
#pragma unroll
                    for (int q = 0; q < 16; ++q) acc[c0 + q] += __uint_as_float(v[q]);
                }
            }
            tc::fence_before_sync();
            __syncwarp();
            if (lane == 0) tc::mbar_arrive_cluster(tc::mapa(tc::smem_u32(&acce[b]), 0));
        }
    }
    __syncwarp();
    // both CTAs of the pair take the same outcome: either one's failure
    const bool mine = __syncthreads_and(good && !*abort_flag) != 0;
    if (!mine && threadIdx.x == 0) tc::st_cluster_u32(tc::mapa(tc::smem_u32((const void *)abort_flag), rank ^ 1u), 1u);
    __syncwarp();
    tc::cluster_sync();
    const bool all_good = mine && !*abort_flag;
    if (!all_good) {
        // the copies already issued land before the ring is used or the CTA
        // exits; they count on the leader's barriers, of which an abort may
        // leave some unarmed, so both CTAs wait by the clock
        if (threadIdx.x == 0) tc::wait_ns(100000000ull);
        __syncthreads();
    }

    // ---------------- epilogue (drain warps) ----------------
    // Each drain warp owns a 32-row x 128-column piece, in 128-row block ib and
    // 128-column block jb of the matrix.  Symmetric product: jb < ib is added
    // and mirrored, jb == ib (the diagonal block) is added in full, jb > ib lies
    // above the diagonal and is left to the CTA that holds its mirror image (a
    // swapped tile lies above it as a whole and is added mirrored).
    // (The sums leave their registers here at once: with both directions written
    // from registers the kernel spilled 388 bytes a thread, in the drain loop too:
    // n = 2056, T = 50,001 with D 661 us, 568 without.)
    if (warp < DRAIN_WARPS && (nk > 0 || !all_good)) {
        const bool direct = part == nullptr;
        const int ib = 2 * tl.ti + (int)rank, jb = 2 * tl.tj + (warp >> 2);
        const bool plain = tl.cross ? !tl.swap : (tl.swap ? direct : jb <= ib);              // at [i][j]
        const bool turned = tl.cross ? tl.swap : (tl.swap || (direct && jb < ib));           // at [j][i]
        const float mul = tl.cross ? sign : 1.f, nan = __int_as_float(0x7fc00000);
        float *o1 = direct ? H : (tl.cross ? partC : part) + (int64_t)blockIdx.y * n * n;
        float *o2 = direct && !tl.cross ? H2 : nullptr;
        float *st = reinterpret_cast<float *>(smem) + warp * 32 * 33;
        const int64_t gi0 = i0 + (warp & 3) * 32, gi = gi0 + lane;
#pragma unroll
        for (int c0 = 0; c0 < 128; c0 += 32) {
            const int64_t gj0 = (int64_t)tl.tj * TN + (warp >> 2) * 128 + c0;
            if (gj0 >= n || gi0 >= n) continue;
#pragma unroll
            for (int q = 0; q < 32; ++q) st[lane * 33 + q] = mul * acc[c0 + q];
            __syncwarp();
#pragma unroll 1
            for (int w = 0; w < 2; ++w) {
                float *o = w ? o2 : o1;
                if (!o) break;
                // 32 x 16 of the piece at a time: its old values first
                auto add = [&](float *d, int64_t at, const float *src, int step) {
#pragma unroll 1
                    for (int h = 0; h < 32; h += 16, d += 16 * n, at += 16, src += 16 * step) {
                        float old[16];
#pragma unroll
                        for (int q = 0; q < 16; ++q) old[q] = direct && at + q < n ? d[q * n] : 0.f;
#pragma unroll
                        for (int q = 0; q < 16; ++q)
                            if (at + q < n) d[q * n] = all_good ? old[q] + src[q * step] : nan;
                    }
                };
                if (turned && gi < n) add(o + gj0 * n + gi, gj0, st + lane * 33, 1);
                if (plain && gj0 + lane < n) add(o + gi0 * n + gj0 + lane, gi0, st + lane, 33);
            }
            __syncwarp();
        }
    }
    if (!all_good && threadIdx.x == 0 && err) atomicOr(err, ST_TIMEOUT);
    tc::fence_before_sync();
    __syncthreads();
    tc::cluster_sync();   // neither CTA leaves while the other may signal its barriers
    if (warp == 0) tc::tmem_dealloc_pair(tmem, 2 * TN);
}

// s += a with the rounding error kept in e
__device__ __forceinline__ void two_sum(float &s, float &e, float a) {
    const float t = s + a, z = t - s;
    e += (s - (t - z)) + (a - z);
    s = t;
}

// H += the symmetric partial sums over the splits, mirrored, and with D also
// D += symmetric - cross partial sums.  One CTA per TILE x TILE tile (bi >= bj)
// of the lower triangle, four columns per thread with all splits' loads in
// flight; the mirror image goes through shared memory, so that every access is
// part of a row of float4 (n a multiple of 8; the caller's H and D, of which
// only 4-byte alignment is asked, go word by word where either has no 16-byte
// base: VEC false).  Sums carry their rounding error: D is the small difference
// of two large sums.  MS bounds the splits (4, 8 or 16), so that few splits take
// few registers.
constexpr int MAX_SPLITS = 16;
template <bool VEC>
__device__ __forceinline__ float4 row4(const float *p) {
    return VEC ? *reinterpret_cast<const float4 *>(p) : make_float4(p[0], p[1], p[2], p[3]);
}
template <bool VEC>
__device__ __forceinline__ void put4(float *p, float4 v) {
    if (VEC) {
        *reinterpret_cast<float4 *>(p) = v;
    } else {
        p[0] = v.x;
        p[1] = v.y;
        p[2] = v.z;
        p[3] = v.w;
    }
}
template <bool CROSS, int MS, int TILE, bool VEC>
__global__ void __launch_bounds__(256) hess_tc_reduce_kernel(int64_t n, int splits, const float *part,
                                                             const float *partC, float *H, float *D) {
    constexpr int TPR = TILE / 4, ROWS = 256 / TPR, PER = TILE / ROWS;   // threads per row, rows per pass, passes
    __shared__ float th[TILE][TILE + 1], tl[TILE][TILE + 1];
    int bi = (int)((sqrt(8.0 * (double)blockIdx.x + 1.0) - 1.0) * 0.5);
    while ((int64_t)(bi + 1) * (bi + 2) / 2 <= blockIdx.x) ++bi;
    while ((int64_t)bi * (bi + 1) / 2 > blockIdx.x) --bi;
    const int bj = (int)(blockIdx.x - (int64_t)bi * (bi + 1) / 2);
    const int r0 = threadIdx.x / TPR, c = (threadIdx.x % TPR) * 4;
    const int64_t nn = n * n;
    auto sum = [&](const float *p, float (&s)[4], float (&e)[4]) {
        float4 v[MS];
#pragma unroll
        for (int k = 0; k < MS; ++k)
            if (k < splits) v[k] = *reinterpret_cast<const float4 *>(p + k * nn);
#pragma unroll
        for (int k = 0; k < MS; ++k)
            if (k < splits) {
                two_sum(s[0], e[0], v[k].x); two_sum(s[1], e[1], v[k].y);
                two_sum(s[2], e[2], v[k].z); two_sum(s[3], e[3], v[k].w);
            }
    };
    auto add = [&](int64_t at, const float (&s)[4], const float (&e)[4]) {
        if (CROSS) {
            float x[4] = {}, xe[4] = {};
            sum(partC + at, x, xe);
            float4 d = row4<VEC>(D + at);
            d.x += (s[0] - x[0]) + (e[0] - xe[0]);
            d.y += (s[1] - x[1]) + (e[1] - xe[1]);
            d.z += (s[2] - x[2]) + (e[2] - xe[2]);
            d.w += (s[3] - x[3]) + (e[3] - xe[3]);
            put4<VEC>(D + at, d);
        }
        float4 h = row4<VEC>(H + at);
        h.x += s[0] + e[0]; h.y += s[1] + e[1]; h.z += s[2] + e[2]; h.w += s[3] + e[3];
        put4<VEC>(H + at, h);
    };
#pragma unroll
    for (int u = 0; u < PER; ++u) {
        const int r = r0 + u * ROWS;
        const int64_t i = (int64_t)bi * TILE + r, j = (int64_t)bj * TILE + c;
        float s[4] = {}, e[4] = {};
        if (i < n && j < n) {
            sum(part + i * n + j, s, e);
            add(i * n + j, s, e);
        }
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            th[r][c + q] = s[q];
            tl[r][c + q] = e[q];
        }
    }
    if (bi == bj) return;
    __syncthreads();
#pragma unroll
    for (int u = 0; u < PER; ++u) {
        const int r = r0 + u * ROWS;
        const int64_t i = (int64_t)bj * TILE + r, j = (int64_t)bi * TILE + c;
        if (i >= n || j >= n) continue;
        float s[4], e[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            s[q] = th[c + q][r];
            e[q] = tl[c + q][r];
        }
        add(i * n + j, s, e);
    }
}

using EncodeFn = CUresult (*)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *,
                              const cuuint64_t *, const cuuint32_t *, const cuuint32_t *, CUtensorMapInterleave,
                              CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
EncodeFn g_encode = nullptr;
std::once_flag g_encode_once;

}  // namespace

static CUresult encode_tmap_2d(CUtensorMapDataType dt, CUtensorMap *map, const void *base, uint64_t inner,
                               uint64_t outer, uint64_t row_stride_bytes, uint32_t box_inner, uint32_t box_outer,
                               int swizzle128);

CUresult encode_tmap_2d_bf16(CUtensorMap *map, const void *base, uint64_t inner, uint64_t outer,
                             uint64_t row_stride_bytes, uint32_t box_inner, uint32_t box_outer, int swizzle128) {
    return encode_tmap_2d(CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, map, base, inner, outer, row_stride_bytes, box_inner,
                          box_outer, swizzle128);
}

CUresult encode_tmap_2d_f32(CUtensorMap *map, const void *base, uint64_t inner, uint64_t outer,
                            uint64_t row_stride_bytes, uint32_t box_inner, uint32_t box_outer, int swizzle128) {
    return encode_tmap_2d(CU_TENSOR_MAP_DATA_TYPE_FLOAT32, map, base, inner, outer, row_stride_bytes, box_inner,
                          box_outer, swizzle128);
}

static bool load_encode() {
    std::call_once(g_encode_once, [] {
        void *fn = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &fn, 12000, cudaEnableDefault, &q) ==
                cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            g_encode = reinterpret_cast<EncodeFn>(fn);
    });
    return g_encode != nullptr;
}

static CUresult encode_tmap_2d(CUtensorMapDataType dt, CUtensorMap *map, const void *base, uint64_t inner,
                               uint64_t outer, uint64_t row_stride_bytes, uint32_t box_inner, uint32_t box_outer,
                               int swizzle128) {
    if (!load_encode()) return CUDA_ERROR_NOT_FOUND;
    cuuint64_t dims[2] = {inner, outer};
    cuuint64_t strides[1] = {row_stride_bytes};
    cuuint32_t box[2] = {box_inner, box_outer};
    cuuint32_t estr[2] = {1, 1};
    return g_encode(map, dt, 2, const_cast<void *>(base), dims, strides, box, estr,
                    CU_TENSOR_MAP_INTERLEAVE_NONE,
                    swizzle128 == 2 ? CU_TENSOR_MAP_SWIZZLE_64B
                                    : (swizzle128 ? CU_TENSOR_MAP_SWIZZLE_128B : CU_TENSOR_MAP_SWIZZLE_NONE),
                    CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
}

CUresult encode_tmap_3d_bf16(CUtensorMap *map, const void *base, uint64_t inner, uint64_t outer, uint64_t planes,
                             uint64_t row_stride_bytes, uint64_t plane_stride_bytes, uint32_t box_inner,
                             uint32_t box_outer, uint32_t box_planes) {
    if (!load_encode()) return CUDA_ERROR_NOT_FOUND;
    cuuint64_t dims[3] = {inner, outer, planes};
    cuuint64_t strides[2] = {row_stride_bytes, plane_stride_bytes};
    cuuint32_t box[3] = {box_inner, box_outer, box_planes};
    cuuint32_t estr[3] = {1, 1, 1};
    return g_encode(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void *>(base), dims, strides, box, estr,
                    CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_64B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                    CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
}

CUresult encode_tmap_2d_f16(CUtensorMap *map, const void *base, uint64_t inner, uint64_t outer,
                            uint64_t row_stride_bytes, uint32_t box_inner, uint32_t box_outer, int swizzle) {
    return encode_tmap_2d(CU_TENSOR_MAP_DATA_TYPE_FLOAT16, map, base, inner, outer, row_stride_bytes, box_inner,
                          box_outer, swizzle);
}

bool hessian_tc_eligible(int64_t n, int64_t T, const void *X) {
    return n >= 64 && n % 8 == 0 && (reinterpret_cast<uintptr_t>(X) & 15) == 0 && T > 0 && T < (1ll << 31) &&
           n < (1ll << 31);
}

// Token splits of a launch of full (and, as 0.35 of one, last-block) tiles over
// the pairs of SMs: the count that minimises rounds x (a split's share of a
// tile's time + a CTA's fixed cost) + the partial sums' traffic, in microseconds
// (a 64-token stage of a pair is 0.29 us at 1.75 GHz; a CTA's start, fill and
// epilogue about 8 us; a partial 256 x 256 tile written and read at 5 TB/s).  0.35
// is the time of a last block of 8 channels; a wide one (n % 256 near 256) takes
// up to a full tile's time, which the count then undercharges (n = 2040, T =
// 50,001 takes 197 us so, against 344 on the kernel before the pairs).  At least
// 1024 tokens per split and at most 16 splits.
static int tc_splits(const HessGrid &g, int64_t T, int sms) {
    const int64_t full = (g.nsym ? (int64_t)g.nf * (g.nf + 1) / 2 : 0) + (g.ncross ? (int64_t)g.nf * g.nf : 0);
    const double tiles = (double)full + 0.35 * (double)(g.nsym + g.ncross - full);
    const int pairs = sms / 2 > 0 ? sms / 2 : 1;
    const int64_t most = std::min<int64_t>(MAX_SPLITS, std::max<int64_t>(1, T / 1024));
    double best = 1e300;
    int bs = 1;
    for (int k = 1; k <= most; ++k) {
        const double rounds = std::ceil(tiles * k / pairs - 1e-9);
        const double us = rounds * ((double)T / 64.0 * 0.29 / k + 8.0) + (k > 1 ? k * tiles * 0.105 : 0.0);
        if (us < best * (1.0 - 1e-9)) {
            best = us;
            bs = k;
        }
    }
    return bs;
}

size_t hessian_tc_ws_bytes(int64_t n, int64_t T, bool cross, int sms) {
    const int k = tc_splits(hess_grid(n, true, false), T, sms);
    return k > 1 ? (size_t)k * n * n * sizeof(float) * (cross ? 2 : 1) : 0;
}

// H += X_Aᵀ X_B (symmetric; X_B null: X_A) when H is given, and D += sign (...):
// with X_C, cross tiles X_Cᵀ X_B.  H and D with X_C: H += X_Aᵀ X_A, D += that
// - X_Cᵀ X_A.
static realq_status_t hess_tc_launch(cudaStream_t s, int64_t n, int64_t T, const void *XA, const void *XB,
                                     const void *XC, float *H, float *D, int *err, void *ws, size_t ws_bytes, int sms,
                                     const char *name, int chunk_stages) {
    CUtensorMap mapA, mapB, mapC;
    CUresult cr = CUDA_SUCCESS;
    auto map = [&](CUtensorMap *m, const void *X) {
        if (cr == CUDA_SUCCESS)
            cr = encode_tmap_2d_bf16(m, X, (uint64_t)n, (uint64_t)T, (uint64_t)n * 2, 64, KSTAGE, 1);
    };
    map(&mapA, XA);
    map(&mapB, XB ? XB : XA);
    map(&mapC, XC ? XC : XA);
    if (cr != CUDA_SUCCESS) return fail(REALQ_ERR_CUDA, "cuTensorMapEncodeTiled failed (%d)", (int)cr);
    // the symmetric product's count also with cross tiles, by the room for its
    // own partial sums: H then has the same bits whether or not D is asked for,
    // whatever the workspace
    const size_t per = (size_t)n * n * sizeof(float);
    int splits = tc_splits(hess_grid(n, true, false), T, sms);
    if (splits > 1 && (ws == nullptr || ws_bytes < 2 * per)) splits = 1;
    if (splits > 1 && (size_t)splits * per > ws_bytes) splits = (int)(ws_bytes / per);   // (at most the plan's)
    int64_t tper = (T + splits - 1) / splits;
    tper = (tper + KSTAGE - 1) / KSTAGE * KSTAGE;
    splits = (int)((T + tper - 1) / tper);
    REALQ_TRY(set_smem_limit(reinterpret_cast<const void *>(hess_tc_kernel), SMEM_BYTES));
    float *part = splits > 1 ? static_cast<float *>(ws) : nullptr;
    // both products' partial sums side by side where the workspace holds them,
    // else one after the other
    const bool both = XC && 2 * (size_t)splits * per <= ws_bytes;
    float *partC = both ? part + (size_t)splits * n * n : part;
    auto launch = [&](const HessGrid &g, float *o, float *o2, float sign, const char *who) -> realq_status_t {
        cudaLaunchConfig_t cfg{};
        cfg.gridDim = dim3((unsigned)(2 * (g.nsym + g.ncross)), (unsigned)splits);
        cfg.blockDim = dim3(THREADS);
        cfg.dynamicSmemBytes = SMEM_BYTES;
        cfg.stream = s;
        cudaLaunchAttribute at[1];
        at[0].id = cudaLaunchAttributeClusterDimension;
        at[0].val.clusterDim.x = 2;
        at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
        cfg.attrs = at;
        cfg.numAttrs = 1;
        {
            Launch L(who, s);
            REALQ_CUDA_TRY(cudaLaunchKernelEx(&cfg, hess_tc_kernel, mapA, mapB, mapC, g, T, tper, o, o2, part, partC,
                                              sign, chunk_stages, err));
        }
        return check_launch(who);
    };
    if (!part) {
        // one split: straight into H and D
        REALQ_TRY(launch(hess_grid(n, true, false), H, XC ? D : nullptr, 1.f, name));
        if (XC) REALQ_TRY(launch(hess_grid(n, false, true), D, nullptr, -1.f, "hessian_cross_tc"));
        return REALQ_OK;
    }
    REALQ_TRY(launch(hess_grid(n, true, both), nullptr, nullptr, 1.f, name));
    const bool vec = ((reinterpret_cast<uintptr_t>(H) | (XC ? reinterpret_cast<uintptr_t>(D) : 0)) & 15) == 0;
    // 64 x 64 tiles where they fill the SMs twice over, else 32 x 32 (n = 1024:
    // 136 tiles took 24 us, 528 take 11)
    const int tile = vec && n >= 1536 ? 64 : 32;
    const int64_t nb = ceil_div(n, tile);
    const unsigned tiles = (unsigned)(nb * (nb + 1) / 2);
    auto reduce = [&](auto cross, auto ms, float *h) {
        constexpr bool CR = decltype(cross)::value;
        constexpr int MS = decltype(ms)::value;
        if (!vec) hess_tc_reduce_kernel<CR, MS, 32, false><<<tiles, 256, 0, s>>>(n, splits, part, partC, h, D);
        else if (tile == 64) hess_tc_reduce_kernel<CR, MS, 64, true><<<tiles, 256, 0, s>>>(n, splits, part, partC, h, D);
        else hess_tc_reduce_kernel<CR, MS, 32, true><<<tiles, 256, 0, s>>>(n, splits, part, partC, h, D);
    };
    auto by_splits = [&](auto cross, float *h) -> realq_status_t {
        {
            Launch L("hessian_reduce", s);
            if (splits <= 4) reduce(cross, std::integral_constant<int, 4>(), h);
            else if (splits <= 8) reduce(cross, std::integral_constant<int, 8>(), h);
            else reduce(cross, std::integral_constant<int, MAX_SPLITS>(), h);
        }
        return check_launch("hessian_reduce");
    };
    if (both) return by_splits(std::true_type(), H);
    REALQ_TRY(by_splits(std::false_type(), H));
    if (!XC) return REALQ_OK;
    REALQ_TRY(by_splits(std::false_type(), D));
    REALQ_TRY(launch(hess_grid(n, false, true), nullptr, nullptr, -1.f, "hessian_cross_tc"));
    return hessian_reduce(s, n, splits, partC, D, 1);
}

realq_status_t hessian_syrk_tc(cudaStream_t s, int64_t n, int64_t T, const void *X, const void *Xfp, float *H, float *D,
                               int *err, void *ws, size_t ws_bytes, int sms) {
    return hess_tc_launch(s, n, T, X, nullptr, Xfp, H, D, err, ws, ws_bytes, sms, "hessian_syrk_tc", CHUNK_STAGES);
}

realq_status_t hessian_pair_tc(cudaStream_t s, int64_t n, int64_t T, const void *XA, const void *XB, float *H, int *err,
                               void *ws, size_t ws_bytes, int sms, int chunk_stages) {
    return hess_tc_launch(s, n, T, XA, XB, nullptr, H, nullptr, err, ws, ws_bytes, sms, "hessian_weighted_tc",
                          chunk_stages);
}

}  // namespace realq

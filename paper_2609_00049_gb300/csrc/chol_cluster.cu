// The factor of a diagonal block of up to 512 columns in one launch: with
// Hd = R R^T (R upper, Cholesky from the last index backwards), U = R^-1 of
// the block, in place, by one thread-block cluster.
//
// The chain through the block's 64-wide pieces is serial: factor piece K,
// solve its panel, update the next diagonal piece.  As separate launches each
// step paid for five to nine kernels and their events (about 50 us a step at
// n = 1024).  Here CTA 0 runs the chain
// and the other CTAs of the cluster everything else (the panel's other rows,
// the trailing updates, the row blocks of U), one step behind it; hardware
// cluster barriers order the steps, and the block itself stays in L2.
//
//   step K (from the last piece to the first):
//     CTA 0    factor and invert piece K in shared memory (V = U_KK)
//     -- barrier 1: V and the updates of step K + 1 are in memory --
//     CTA c    panel R[i, K] = A[i, K] V^T for i = K - 1 - c
//     -- barrier 2: the panel is in memory (CTA 0 only arrives) --
//     CTA 0    its own update A[K-1, K-1] -= R[K-1, K] R[K-1, K]^T, and on
//              to piece K - 1
//     others   A[i, j] -= R[i, K] R[j, K]^T for the other pairs, and
//              U[K, j] = -V (R[K, K+1:] U[K+1:, j]) in slices of 32 columns,
//              held in shared memory until barrier 1 of the next step, when
//              no other CTA reads R[K, :] any more
//
// All arithmetic is fp32 FFMA with every sum taken in index order.
//
// Measured, 512 columns: 130 us (16 us a step; of its 31 k cycles the two 32 x 32
// factors take 11 k, the panel 5 k, the products inside the piece 4 k, the next
// piece's update 3 k, the barrier and the loads 3.5 k), against about 400 us as
// separate launches.  What bounds it is latency: one SM runs the chain, and a
// pivot costs about 170 cycles of shared-memory round trips, a reciprocal root
// and dependent FMAs.
#include "kernels.cuh"

#include <map>
#include <mutex>
#include <utility>

namespace realq {
namespace {

constexpr int NB = 64;
constexpr int TH = 256;
constexpr int P = 68;             // pitch of an operand's rows (float4 along the row, rows 4 banks apart)
constexpr int MAX_HOLD = 2;       // slices of U's row block that a CTA may hold over a barrier
constexpr int SL = 32;            // columns of a slice

// The products below are bound by what shared memory delivers (32 floats per
// cycle and SM, broadcast or not) before the FMA pipe, so each thread takes
// 8 x 4 or 4 x 4 outputs and reads four terms of a row at a time.
struct __align__(16) Sm {
    float A[NB * P];              // operand rows [i][k]
    float B[NB * P];              // operand rows [j][k], or [k][j] in u_slice; CTA 0: V
    float hold[MAX_HOLD][NB * SL];
    float S11[32][33], S22[32][33];
    __align__(16) float A12[32][36];
    __align__(16) float R12[32][36];
    __align__(16) float X[32][36];
    __align__(16) float bc[2][4][32];
    __align__(16) float bv[2][4][32];
    __align__(16) float rinv[32];
};

__device__ __forceinline__ void cluster_arrive() {
    __syncwarp();
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
}
__device__ __forceinline__ void cluster_wait() {
    __syncwarp();
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// a 64 x 64 block of which rows x cols exist (zeros elsewhere): 16 values per
// thread, row (t / 16) + 16 u, columns (t % 16) * 4 ..
template <bool VEC>
__device__ __forceinline__ void fetch(float4 (&v)[4], const float *src, int64_t ld, int rows, int cols) {
    const int r0 = threadIdx.x >> 4, c = (threadIdx.x & 15) * 4;
#pragma unroll
    for (int u = 0; u < 4; ++u) {
        const int r = r0 + 16 * u;
        const float *s = src + r * ld + c;
        v[u] = make_float4(0.f, 0.f, 0.f, 0.f);
        if (r < rows) {
            if (VEC && c + 3 < cols) {
                v[u] = __ldcg(reinterpret_cast<const float4 *>(s));
            } else {
                if (c < cols) v[u].x = __ldcg(s);
                if (c + 1 < cols) v[u].y = __ldcg(s + 1);
                if (c + 2 < cols) v[u].z = __ldcg(s + 2);
                if (c + 3 < cols) v[u].w = __ldcg(s + 3);
            }
        }
    }
}
__device__ __forceinline__ void stash(float *dst, const float4 (&v)[4]) {
    const int r0 = threadIdx.x >> 4, c = (threadIdx.x & 15) * 4;
#pragma unroll
    for (int u = 0; u < 4; ++u) *reinterpret_cast<float4 *>(dst + (r0 + 16 * u) * P + c) = v[u];
}

// acc[p][q] = sum_k A[ty + SY p][k] B[tx + SX q][k] over K terms, in order
// (the next four terms are read while the current ones are multiplied: with
// one or two warps per scheduler nothing else hides the latency)
template <int PR, int QC, int SY, int SX, int K, int PA, int PBT>
__device__ __forceinline__ void mma_nt(const float *A, const float *B, int ty, int tx, float (&acc)[PR][QC]) {
#pragma unroll
    for (int p = 0; p < PR; ++p)
#pragma unroll
        for (int q = 0; q < QC; ++q) acc[p][q] = 0.f;
    float4 a[2][PR], b[2][QC];
    auto load = [&](int k, int s) {
#pragma unroll
        for (int q = 0; q < QC; ++q) b[s][q] = *reinterpret_cast<const float4 *>(B + (tx + SX * q) * PBT + k);
#pragma unroll
        for (int p = 0; p < PR; ++p) a[s][p] = *reinterpret_cast<const float4 *>(A + (ty + SY * p) * PA + k);
    };
    load(0, 0);
#pragma unroll 1
    for (int k = 0; k < K; k += 8) {
#pragma unroll
        for (int s = 0; s < 2; ++s) {
            load((k + 4 * s + 4) & (K - 1), s ^ 1);   // (the last one wraps around and is not used)
#pragma unroll
            for (int e = 0; e < 4; ++e)
#pragma unroll
                for (int p = 0; p < PR; ++p) {
                    const float4 &u = a[s][p];
                    const float av = e == 0 ? u.x : e == 1 ? u.y : e == 2 ? u.z : u.w;
#pragma unroll
                    for (int q = 0; q < QC; ++q) {
                        const float4 &w = b[s][q];
                        acc[p][q] = fmaf(av, e == 0 ? w.x : e == 1 ? w.y : e == 2 ? w.z : w.w, acc[p][q]);
                    }
                }
        }
    }
}

// acc[p][q] += sum_k A[ty + SY p][k] B[k][4 tx + q] over K terms, in order
template <int SY, int K, int PA, int PBN>
__device__ __forceinline__ void mma_nn(const float *A, const float *B, int ty, int tx, float (&acc)[4][4]) {
    float4 a[2][4], b[2][4];
    auto load = [&](int k, int s) {
#pragma unroll
        for (int p = 0; p < 4; ++p) a[s][p] = *reinterpret_cast<const float4 *>(A + (ty + SY * p) * PA + k);
#pragma unroll
        for (int e = 0; e < 4; ++e) b[s][e] = *reinterpret_cast<const float4 *>(B + (k + e) * PBN + tx * 4);
    };
    load(0, 0);
#pragma unroll 1
    for (int k = 0; k < K; k += 8) {
#pragma unroll
        for (int s = 0; s < 2; ++s) {
            load((k + 4 * s + 4) & (K - 1), s ^ 1);
#pragma unroll
            for (int e = 0; e < 4; ++e)
#pragma unroll
                for (int p = 0; p < 4; ++p) {
                    const float av = e == 0 ? a[s][p].x : e == 1 ? a[s][p].y : e == 2 ? a[s][p].z : a[s][p].w;
                    acc[p][0] = fmaf(av, b[s][e].x, acc[p][0]);
                    acc[p][1] = fmaf(av, b[s][e].y, acc[p][1]);
                    acc[p][2] = fmaf(av, b[s][e].z, acc[p][2]);
                    acc[p][3] = fmaf(av, b[s][e].w, acc[p][3]);
                }
        }
    }
}

// A 32 x 32 piece S (upper triangle): reverse-order Cholesky S = R R^T fused
// with the back substitution V = R^-1 (zeros below the diagonal), 256 threads;
// V[r * P + c].  Lane j owns column j of the piece (warps 0-3, eight rows each)
// and row j of V (warps 4-7, eight entries each), in registers.  Pivots go four
// at a time: their columns and V rows are published (unscaled) in a
// double-buffered slot with one barrier, and every thread repeats the 4 x 4
// elimination among them for the entries that it needs, so the chain pays one
// barrier per four pivots; a warp whose rows lie below the pivots (or whose V
// entries are still zero) only meets the barrier.  Each entry receives
// a_ij -= r_ik r_jk, V[j] -= r_jk V[k] pivot by pivot in descending order, as
// with one pivot at a time (entries below the diagonal take part and are never
// read).  A pivot that is not positive (or not finite) is recorded (the first
// one wins; columns >= valid are padding) and replaced by 1 to keep going.
__device__ __forceinline__ void rchol_inv32(const float (*S)[33], float *V, float (*bc)[4][32], float (*bv)[4][32],
                                            float *rinvs, int *status, int64_t col0, int valid) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, q0 = (warp & 3) * 8;
    const bool isv = warp >= 4;
    float (*own)[4][32] = isv ? bv : bc;
    float x[8];
#pragma unroll
    for (int q = 0; q < 8; ++q) x[q] = isv ? (q0 + q == lane ? 1.f : 0.f) : S[q0 + q][lane];
    int first = -1;
#pragma unroll 1
    for (int g = 7; g >= 0; --g) {
        const int p = 4 * g, b = g & 1;
        if (lane >= p && lane < p + 4) {
            *reinterpret_cast<float4 *>(&own[b][lane - p][q0]) = make_float4(x[0], x[1], x[2], x[3]);
            *reinterpret_cast<float4 *>(&own[b][lane - p][q0 + 4]) = make_float4(x[4], x[5], x[6], x[7]);
        }
        __syncthreads();
        if (isv ? q0 + 7 < p : q0 > p + 3) continue;
        // the elimination among the four pivots: rinv[s] = 1 / r of pivot
        // p + s and cf[s][t] the factor of column p + t against it.  A
        // normal positive pivot takes the hardware's reciprocal root as it
        // stands; with any other the four are done again with the checks
        float D[4][4], rinv[4], cf[4][4];
        bool plain = true;
        auto head = [&](auto root) {
#pragma unroll
            for (int s = 0; s < 4; ++s) {
                const float4 d = *reinterpret_cast<const float4 *>(&bc[b][s][p]);
                D[s][0] = d.x; D[s][1] = d.y; D[s][2] = d.z; D[s][3] = d.w;
            }
#pragma unroll
            for (int s = 3; s >= 0; --s) {
                rinv[s] = root(s, D[s][s]);
#pragma unroll
                for (int t = s - 1; t >= 0; --t) {
                    const float rt = D[s][t] * rinv[s];
                    cf[s][t] = -rt * rinv[s];
#pragma unroll
                    for (int u = 0; u <= t; ++u) D[t][u] = fmaf(D[s][u], cf[s][t], D[t][u]);
                }
            }
        };
        head([&](int, float d) {
            float r;
            asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(d));
            plain = plain && d >= 1.17549435e-38f && d < __int_as_float(0x7f800000);
            return r;
        });
        float ar[4][8], al[4];
#pragma unroll
        for (int s = 3; s >= 0; --s) {
            const float4 a0 = *reinterpret_cast<const float4 *>(&own[b][s][q0]);
            const float4 a1 = *reinterpret_cast<const float4 *>(&own[b][s][q0 + 4]);
            ar[s][0] = a0.x; ar[s][1] = a0.y; ar[s][2] = a0.z; ar[s][3] = a0.w;
            ar[s][4] = a1.x; ar[s][5] = a1.y; ar[s][6] = a1.z; ar[s][7] = a1.w;
            al[s] = bc[b][s][lane];
        }
        if (!plain)
            head([&](int s, float d) {
                const bool bad = !(d > 0.f) || !isfinite(d);
                if (bad && first < 0 && p + s < valid) first = p + s;
                return rsqrtf(bad ? 1.f : d);
            });
        if (threadIdx.x == 0) *reinterpret_cast<float4 *>(rinvs + p) = make_float4(rinv[0], rinv[1], rinv[2], rinv[3]);
#pragma unroll
        for (int s = 3; s >= 0; --s) {
            const float rjk = lane < p + s ? al[s] * rinv[s] : 0.f;
            const float cx = -rjk * rinv[s];
#pragma unroll
            for (int t = s - 1; t >= 0; --t) {
                al[t] = fmaf(al[s], cf[s][t], al[t]);
#pragma unroll
                for (int q = 0; q < 8; ++q) ar[t][q] = fmaf(ar[s][q], cf[s][t], ar[t][q]);
            }
#pragma unroll
            for (int q = 0; q < 8; ++q) x[q] = fmaf(ar[s][q], cx, x[q]);
        }
    }
    __syncthreads();
    if (isv) {
        const float rown = rinvs[lane];
        *reinterpret_cast<float4 *>(V + lane * P + q0) = make_float4(x[0] * rown, x[1] * rown, x[2] * rown, x[3] * rown);
        *reinterpret_cast<float4 *>(V + lane * P + q0 + 4) =
            make_float4(x[4] * rown, x[5] * rown, x[6] * rown, x[7] * rown);
    }
    if (threadIdx.x == 0 && first >= 0) atomicCAS(status, -1, (int)(col0 + first));
    __syncthreads();
}

// Piece [k0, k0 + kb) from S11 / A12 / S22 (split 2 x 2 into 32 x 32):
//   A22 = R22 R22^T,  R12 = A12 R22^-T,  A11 - R12 R12^T = R11 R11^T,
//   V = R^-1 = [[V11, -V11 R12 V22], [0, V22]].
// V goes to A (upper, in place of the piece) and to sm.B (rows, zeros below).
__device__ __forceinline__ void factor_piece(Sm &sm, float *A, int64_t ld, int kb, int *status, int64_t col0) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    float *V = sm.B, *V22 = sm.B + 32 * P + 32;
    const int tx = lane & 7, ty = (lane >> 3) + 4 * (warp & 1);   // 32 x 32 outputs over a warp pair
    // the quarter below the diagonal
    for (int e = threadIdx.x; e < 32 * 32; e += TH) V[(32 + (e >> 5)) * P + (e & 31)] = 0.f;
    rchol_inv32(sm.S22, V22, sm.bc, sm.bv, sm.rinv, status, col0 + 32, kb - 32);
    if (warp < 2) {
        // R12[i][j] = sum_l A12[i][l] V22[j][l]
        float acc[4][4];
        mma_nt<4, 4, 8, 8, 32, 36, P>(&sm.A12[0][0], V22, ty, tx, acc);
#pragma unroll
        for (int p = 0; p < 4; ++p)
#pragma unroll
            for (int q = 0; q < 4; ++q) sm.R12[ty + 8 * p][tx + 8 * q] = acc[p][q];
    }
    __syncthreads();
    if (warp < 2) {
        // A11 -= R12 R12^T
        float acc[4][4];
        mma_nt<4, 4, 8, 8, 32, 36, 36>(&sm.R12[0][0], &sm.R12[0][0], ty, tx, acc);
#pragma unroll
        for (int p = 0; p < 4; ++p)
#pragma unroll
            for (int q = 0; q < 4; ++q) sm.S11[ty + 8 * p][tx + 8 * q] -= acc[p][q];
    } else if (warp < 4) {
        // X = R12 V22
        float acc[4][4] = {};
        mma_nn<8, 32, 36, P>(&sm.R12[0][0], V22, ty, tx, acc);
#pragma unroll
        for (int p = 0; p < 4; ++p)
            *reinterpret_cast<float4 *>(&sm.X[ty + 8 * p][tx * 4]) = make_float4(acc[p][0], acc[p][1], acc[p][2], acc[p][3]);
    }
    __syncthreads();
    rchol_inv32(sm.S11, V, sm.bc, sm.bv, sm.rinv, status, col0, kb);
    if (warp < 2) {
        // V12 = -V11 X
        float acc[4][4] = {};
        mma_nn<8, 32, P, 36>(V, &sm.X[0][0], ty, tx, acc);
#pragma unroll
        for (int p = 0; p < 4; ++p)
            *reinterpret_cast<float4 *>(V + (ty + 8 * p) * P + 32 + tx * 4) =
                make_float4(-acc[p][0], -acc[p][1], -acc[p][2], -acc[p][3]);
    }
    __syncthreads();
#pragma unroll 4
    for (int u = 0; u < NB * NB / TH; ++u) {
        const int e = threadIdx.x + u * TH, r = e >> 6, c = e & 63;
        if (r < kb && c < kb && c >= r) A[r * ld + c] = V[r * P + c];
    }
}

// the piece to factor (16 values per thread, as fetch leaves them) into S11 /
// A12 / S22: the upper triangle, padded with the identity from kb on
__device__ __forceinline__ void put_piece(Sm &sm, const float4 (&v)[4], int kb) {
    const int r0 = threadIdx.x >> 4, c = (threadIdx.x & 15) * 4;
#pragma unroll
    for (int u = 0; u < 4; ++u) {
        const int i = r0 + 16 * u;
        const float x[4] = {v[u].x, v[u].y, v[u].z, v[u].w};
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int j = c + q;
            const float w = (i < kb && j < kb) ? (j >= i ? x[q] : 0.f) : (i == j ? 1.f : 0.f);
            if (i < 32) {
                if (j < 32) sm.S11[i][j] = w;
                else sm.A12[i][j - 32] = w;
            } else if (j >= 32) {
                sm.S22[i - 32][j - 32] = w;
            }
        }
    }
}

// R[i, K] = A[i, K] V^T: sm.A holds A[i, K], sm.B V; the result goes to o (its
// first cols columns) and, if keep, over sm.A
__device__ __forceinline__ void panel_product(Sm &sm, float *o, int64_t ld, int cols, bool keep) {
    const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
    float acc[8][4];
    if (threadIdx.x < 128) {
        mma_nt<8, 4, 8, 16, NB, P, P>(sm.A, sm.B, ty, tx, acc);
#pragma unroll
        for (int p = 0; p < 8; ++p)
#pragma unroll
            for (int q = 0; q < 4; ++q)
                if (tx + 16 * q < cols) o[(int64_t)(ty + 8 * p) * ld + tx + 16 * q] = acc[p][q];
    }
    __syncthreads();
    if (keep) {
        if (threadIdx.x < 128) {
#pragma unroll
            for (int p = 0; p < 8; ++p)
#pragma unroll
                for (int q = 0; q < 4; ++q) sm.A[(ty + 8 * p) * P + tx + 16 * q] = acc[p][q];
        }
        __syncthreads();
    }
}

template <bool VEC>
__global__ void __launch_bounds__(TH, 1) chol_cluster_kernel(int64_t ld, float *A, int n, int64_t col0, int *status) {
    extern __shared__ __align__(16) unsigned char raw[];
    Sm &sm = *reinterpret_cast<Sm *>(raw);
    const int cta = (int)blockIdx.x, nc = (int)gridDim.x;   // one cluster
    const int nk = (n + NB - 1) / NB;
    auto blk = [&](int i, int j) { return A + (int64_t)i * NB * ld + j * NB; };
    auto ext = [&](int i) { return min(NB, n - i * NB); };

    int held = 0, hold_K = -1;     // slices of U's row block hold_K to be written
    // slice s (0 .. 2 (nk - 1 - K) - 1) of row block K: the long ones first
    auto slice_of = [&](int s, int &j, int &c) {
        j = nk - 1 - s / (NB / SL);
        c = (s % (NB / SL)) * SL;
    };
    auto write_held = [&](int first, int stride) {
        for (int t = 0; t < held; ++t) {
            int j, c;
            slice_of(first + t * stride, j, c);
            float *o = blk(hold_K, j) + c;
            const int rows = ext(hold_K), cols = ext(j) - c;
#pragma unroll
            for (int u = 0; u < NB * SL / TH; ++u) {
                const int e = threadIdx.x + u * TH, r = e / SL, cc = e % SL;
                if (r < rows && cc < cols) o[(int64_t)r * ld + cc] = sm.hold[t][e];
            }
        }
        held = 0;
    };
    // U[K, slice] = -U_KK (R[K, K+1:] U[K+1:, slice]) into hold[t]
    auto u_slice = [&](int K, int s, int t) {
        int j, c;
        slice_of(s, j, c);
        const int rK = ext(K), cols = ext(j) - c;
        const int stx = threadIdx.x & 7, sty = threadIdx.x >> 3;       // 128 threads: rows sty + 16 p, columns 4 stx ..
        float acc[4][4] = {};
        float4 va[4], vb[2];
        auto fetch_b = [&](int k) {
#pragma unroll
            for (int u = 0; u < 2; ++u) {
                const int r = (threadIdx.x >> 3) + 32 * u, cc = (threadIdx.x & 7) * 4;
                const float *src = blk(k, j) + (int64_t)r * ld + c + cc;
                vb[u] = make_float4(0.f, 0.f, 0.f, 0.f);
                if (r < ext(k)) {
                    if (VEC && cc + 3 < cols) {
                        vb[u] = __ldcg(reinterpret_cast<const float4 *>(src));
                    } else {
                        if (cc < cols) vb[u].x = __ldcg(src);
                        if (cc + 1 < cols) vb[u].y = __ldcg(src + 1);
                        if (cc + 2 < cols) vb[u].z = __ldcg(src + 2);
                        if (cc + 3 < cols) vb[u].w = __ldcg(src + 3);
                    }
                }
            }
        };
        fetch<VEC>(va, blk(K, K + 1), ld, rK, ext(K + 1));
        fetch_b(K + 1);
        for (int k = K + 1; k <= j; ++k) {
            __syncthreads();   // the readers of the buffers are done
            stash(sm.A, va);
#pragma unroll
            for (int u = 0; u < 2; ++u)
                *reinterpret_cast<float4 *>(sm.B + ((threadIdx.x >> 3) + 32 * u) * P + (threadIdx.x & 7) * 4) = vb[u];
            __syncthreads();
            if (k < j) {
                fetch<VEC>(va, blk(K, k + 1), ld, rK, ext(k + 1));
                fetch_b(k + 1);
            } else {
                fetch<VEC>(va, blk(K, K), ld, rK, rK);   // U_KK (upper, zeros below)
            }
            if (threadIdx.x < 128) mma_nn<16, NB, P, P>(sm.A, sm.B, sty, stx, acc);
        }
        __syncthreads();
        stash(sm.A, va);
        if (threadIdx.x < 128) {
#pragma unroll
            for (int p = 0; p < 4; ++p)
                *reinterpret_cast<float4 *>(sm.B + (sty + 16 * p) * P + stx * 4) =
                    make_float4(acc[p][0], acc[p][1], acc[p][2], acc[p][3]);
        }
        __syncthreads();
        if (threadIdx.x < 128) {
            float o[4][4] = {};
            mma_nn<16, NB, P, P>(sm.A, sm.B, sty, stx, o);
#pragma unroll
            for (int p = 0; p < 4; ++p)
#pragma unroll
                for (int q = 0; q < 4; ++q) sm.hold[t][(sty + 16 * p) * SL + stx * 4 + q] = -1.f * o[p][q];
        }
    };

    // ------------------------------------------------ CTA 0: the chain ---
    if (cta == 0) {
        {
            // the last piece
            float4 v[4];
            const int kb = ext(nk - 1);
            fetch<VEC>(v, blk(nk - 1, nk - 1), ld, kb, kb);
            put_piece(sm, v, kb);
            __syncthreads();
        }
        for (int K = nk - 1; K >= 0; --K) {
            const int kb = ext(K);
            factor_piece(sm, blk(K, K), ld, kb, status, col0 + (int64_t)K * NB);
            if (K < nk - 1) cluster_wait();    // barrier 2 of step K + 1 (arrived below)
            cluster_arrive();                  // barrier 1
            cluster_wait();
            if (K == 0) break;
            // panel row K - 1, and the next piece's update from it
            {
                float4 va[4], vd[4];
                fetch<VEC>(va, blk(K - 1, K), ld, NB, kb);
                fetch<VEC>(vd, blk(K - 1, K - 1), ld, NB, NB);
                stash(sm.A, va);
                put_piece(sm, vd, NB);
            }
            __syncthreads();
            panel_product(sm, blk(K - 1, K), ld, kb, true);
            cluster_arrive();                  // barrier 2; waited for after the next piece
            // quarters (0, 0), (0, 1), (1, 1) of A[K-1, K-1] -= R R^T, two warps each
            const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, quarter = warp >> 1;
            if (warp < 6) {
                const int ty = (lane >> 3) + (warp & 1) * 16, tx = lane & 7;
                float up[4][4];
                mma_nt<4, 4, 4, 8, NB, P, P>(sm.A + (quarter == 2 ? 32 * P : 0), sm.A + (quarter >= 1 ? 32 * P : 0), ty,
                                             tx, up);
#pragma unroll
                for (int p = 0; p < 4; ++p)
#pragma unroll
                    for (int q = 0; q < 4; ++q) {
                        const int i = ty + 4 * p, j = tx + 8 * q;
                        if (quarter == 1) sm.A12[i][j] -= up[p][q];
                        else if (j >= i && quarter == 0) sm.S11[i][j] -= up[p][q];
                        else if (j >= i) sm.S22[i][j] -= up[p][q];
                    }
            }
            __syncthreads();
        }
    } else {
        // ------------------------------------------ the other CTAs ---
        for (int K = nk - 1; K >= 0; --K) {
            cluster_arrive();                  // barrier 1
            cluster_wait();
            if (held) write_held(cta - 1, nc - 1);
            if (K == 0) break;
            const int kb = ext(K);
            // (K <= 7 rows of pieces, and CTA 0 takes the first)
            for (int i = K - 1 - cta; i >= 0; i -= nc - 1) {
                float4 va[4], vb[4];
                fetch<VEC>(va, blk(i, K), ld, NB, kb);
                fetch<VEC>(vb, blk(K, K), ld, kb, kb);      // V = U_KK (upper, zeros below)
                __syncthreads();
                stash(sm.A, va);
                stash(sm.B, vb);
                __syncthreads();
                panel_product(sm, blk(i, K), ld, kb, false);
            }
            cluster_arrive();                  // barrier 2
            cluster_wait();
            // updates of the pieces (i, j), i <= j < K, but (K-1, K-1): the
            // next panel's column first
            const int nup = K * (K + 1) / 2 - 1;
            for (int t = cta - 1; t < nup; t += nc - 1) {
                int j = K - 1, i = t;
                if (t >= K - 1) {
                    int r = t - (K - 1);
                    j = K - 2;
                    while (r > j) {
                        r -= j + 1;
                        --j;
                    }
                    i = r;
                }
                float4 va[4], vb[4];
                fetch<VEC>(va, blk(i, K), ld, NB, kb);
                fetch<VEC>(vb, blk(j, K), ld, NB, kb);
                __syncthreads();
                stash(sm.A, va);
                stash(sm.B, vb);
                __syncthreads();
                if (threadIdx.x < 128) {
                    const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
                    float *o = blk(i, j);
                    float cv[8][4], acc[8][4];
#pragma unroll
                    for (int p = 0; p < 8; ++p)
#pragma unroll
                        for (int q = 0; q < 4; ++q) cv[p][q] = __ldcg(o + (int64_t)(ty + 8 * p) * ld + tx + 16 * q);
                    mma_nt<8, 4, 8, 16, NB, P, P>(sm.A, sm.B, ty, tx, acc);
#pragma unroll
                    for (int p = 0; p < 8; ++p)
#pragma unroll
                        for (int q = 0; q < 4; ++q)
                            if (i != j || tx + 16 * q >= ty + 8 * p)
                                o[(int64_t)(ty + 8 * p) * ld + tx + 16 * q] = cv[p][q] - acc[p][q];
                }
            }
            // row block K of U
            const int ns = (nk - 1 - K) * (NB / SL);
            hold_K = K;
            for (int s = cta - 1; s < ns; s += nc - 1) u_slice(K, s, held++);
        }
    }
    // row block 0 of U, by every CTA, once row block 1 is in memory
    cluster_arrive();
    cluster_wait();
    const int ns = (nk - 1) * (NB / SL);
    hold_K = 0;
    for (int s = cta; s < ns; s += nc) u_slice(0, s, held++);
    cluster_arrive();
    cluster_wait();
    write_held(cta, nc);
}

// CTAs of the cluster: 16 where the current device places such a cluster, else
// 8 (held slices: at most 14 of a row block over 7 CTAs, so 2 each).  The
// permission for more than 8 CTAs and the answer both belong to a device: they
// are set and asked once per device and kernel.
realq_status_t cluster_ctas(const void *fn, int *ctas) {
    int dev = 0;
    REALQ_CUDA_TRY(cudaGetDevice(&dev));
    static std::mutex mu;
    static std::map<std::pair<int, const void *>, int> best;
    std::lock_guard<std::mutex> lk(mu);
    int &b = best[{dev, fn}];
    if (!b) {
        b = 8;
        cudaLaunchConfig_t cfg{};
        cfg.gridDim = dim3(16);
        cfg.blockDim = dim3(TH);
        cfg.dynamicSmemBytes = sizeof(Sm);
        cudaLaunchAttribute at[1];
        at[0].id = cudaLaunchAttributeClusterDimension;
        at[0].val.clusterDim.x = 16;
        at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
        cfg.attrs = at;
        cfg.numAttrs = 1;
        int n = 0;
        if (cudaFuncSetAttribute(fn, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess &&
            cudaOccupancyMaxActiveClusters(&n, fn, &cfg) == cudaSuccess) {
            if (n > 0) b = 16;
        } else {
            cudaGetLastError();
        }
    }
    *ctas = b;
    return REALQ_OK;
}

}  // namespace

realq_status_t chol_inv_block(cudaStream_t s, int64_t ld, float *A, int64_t n, int64_t col0, int *status) {
    if (n <= 0) return REALQ_OK;
    if (n > kCholBlock) return fail(REALQ_ERR_INVALID_ARG, "chol_inv_block: %lld columns", (long long)n);
    const bool vec = ld % 4 == 0 && (reinterpret_cast<uintptr_t>(A) & 15) == 0;
    const void *fn = vec ? reinterpret_cast<const void *>(chol_cluster_kernel<true>)
                         : reinterpret_cast<const void *>(chol_cluster_kernel<false>);
    REALQ_TRY(set_smem_limit(fn, (int)sizeof(Sm)));
    // one piece has no panel, no update and no row of U beside it
    int nc = 1;
    if (n > NB) REALQ_TRY(cluster_ctas(fn, &nc));
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)nc);
    cfg.blockDim = dim3(TH);
    cfg.dynamicSmemBytes = sizeof(Sm);
    cfg.stream = s;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = (unsigned)nc;
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    {
        Launch L("chol_block", s);
        if (vec) REALQ_CUDA_TRY(cudaLaunchKernelEx(&cfg, chol_cluster_kernel<true>, ld, A, (int)n, col0, status));
        else REALQ_CUDA_TRY(cudaLaunchKernelEx(&cfg, chol_cluster_kernel<false>, ld, A, (int)n, col0, status));
    }
    return check_launch("chol_block");
}

}  // namespace realq

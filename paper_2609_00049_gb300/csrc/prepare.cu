// Step a3 (Alg. 1: "Compute ... H and its inverse"): H̄ = H_sum / T, dead
// channels, relative damping, and the upper factor U with Hd^-1 = U^T U.
//
// U is obtained without forming Hd^-1: factor Hd = R R^T with R upper
// triangular (Cholesky taken from the last index backwards), then U = R^-1,
// because Hd^-1 = R^-T R^-1 = U^T U.  Row j of U, scaled by U_jj, is row j of
// the inverse Hessian after the Schur-complement downdates of columns < j,
// which is what the OBS step of Eq. (gptq_update) consumes.
//
// Up to 512 columns one thread-block cluster does the whole factor
// (chol_cluster.cu).  Wider inputs are blocked by 512: the cluster factors and
// inverts each diagonal block, and everything beside it is a product of depth
// 512 with fp32 accuracy on the tensor cores (gemm_x6.cu), spread over three
// streams (prepare_blocked below).  The allocation-free entry point takes the
// same steps on one stream, with blocks as deep as its scratch has room for
// operand planes; beyond that (n > 21824) it keeps 64-wide steps on the CUDA
// cores (prepare_steps).  A pivot that is not positive (or not finite) records
// its column in the workspace status word; prepare reads it once at the end,
// the deferred variant leaves it for realq_prepare_status (a captured step
// reads no host memory).
#include "kernels.cuh"

#include <algorithm>
#include <vector>

namespace realq {
namespace {

constexpr int NB = 64;

// Hbar = H / T, A = its upper triangle with the dead channels' diagonal set to
// 1 (zeros below), dead.  Bound by memory (12 bytes per element): a grid row per
// matrix row, so that no element pays a 64-bit division, and with VEC four
// columns per thread (n = 14336: 711 us one element per thread).
template <bool VEC>
__global__ void __launch_bounds__(256) prep_init_kernel(int64_t n, float Tf, const float *H, float *Hbar, float *A,
                                                        uint8_t *dead) {
    const int64_t j0 = ((int64_t)blockIdx.x * 256 + threadIdx.x) * (VEC ? 4 : 1);
    if (j0 >= n) return;
    for (int64_t i = blockIdx.y; i < n; i += gridDim.y) {
        const int64_t at = i * n + j0;
        float h[4], a[4];
        if (VEC) {
            const float4 v = *reinterpret_cast<const float4 *>(H + at);
            h[0] = v.x; h[1] = v.y; h[2] = v.z; h[3] = v.w;
        } else {
            h[0] = H[at];
        }
#pragma unroll
        for (int q = 0; q < (VEC ? 4 : 1); ++q) {
            const int64_t j = j0 + q;
            const bool d = h[q] == 0.f;
            h[q] = h[q] / Tf;
            a[q] = j > i ? h[q] : 0.f;
            if (j == i) {
                dead[i] = d ? 1 : 0;
                a[q] = d ? 1.f : h[q];
            }
        }
        if (VEC) {
            if (Hbar) *reinterpret_cast<float4 *>(Hbar + at) = make_float4(h[0], h[1], h[2], h[3]);
            *reinterpret_cast<float4 *>(A + at) = make_float4(a[0], a[1], a[2], a[3]);
        } else {
            if (Hbar) Hbar[at] = h[0];
            A[at] = a[0];
        }
    }
}

// lambda = damp * mean(diag A) (fp64 reduction in a fixed order); A_jj += lambda
__global__ void prep_damp_kernel(int64_t n, float *A, float damp, float *lam_out) {
    __shared__ double red[1024];
    double s = 0.0;
    for (int64_t j = threadIdx.x; j < n; j += blockDim.x) s += (double)A[j * n + j];
    red[threadIdx.x] = s;
    __syncthreads();
    for (int w = blockDim.x / 2; w > 0; w >>= 1) {
        if ((int)threadIdx.x < w) red[threadIdx.x] += red[threadIdx.x + w];
        __syncthreads();
    }
    const float lam = (float)((double)damp * (red[0] / (double)n));
    for (int64_t j = threadIdx.x; j < n; j += blockDim.x) A[j * n + j] += lam;
    if (threadIdx.x == 0) *lam_out = lam;
}

// A 32 x 32 block As (pitch 33, upper triangle): reverse-order Cholesky
// As = R R^T (R upper) fused with the back substitution V = R^-1, written to
// Vs (row-major, zeros below the diagonal), by the 128 threads of the CTA.
// Lane j owns column j of the block and row j of V; warp w keeps entries
// 8w .. 8w + 7 of both in registers.  Pivot k needs only column k of R and
// row k of V: lane k of every warp publishes its eight entries of both
// (unscaled) into a double-buffered 64-float slot bf[(k & 1) * 64 ..] with
// one CTA barrier per pivot (the slot of pivot k is next written at pivot
// k - 2, after the barrier of pivot k - 1, which every warp reaches only after
// its reads of pivot k); every thread then applies
//   a_ij -= r_ik r_jk (i <= j < k),   V[j] -= r_jk V[k] (j < k),
// with r_ik = a_ik / sqrt(a_kk), to its entries.  Row k of V is scaled by its
// own 1 / r_kk once, at the end (no later pivot reads it).  A pivot that is
// not positive (or not finite) is recorded (the first one wins; columns >=
// valid are padding) and replaced by 1 to keep going.  (One warp doing all 32
// entries issues a ~100-instruction pivot at about seven cycles each; split
// four ways with a barrier the pivot is about three times shorter.)
__device__ __forceinline__ void cta_rchol_inv32(const float (*As)[33], float (*Vs)[33], float *bf, int warp,
                                                int lane, int *status, int64_t col0, int valid) {
    const int q0 = warp * 8;
    float c[8], v[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        c[i] = As[q0 + i][lane];
        v[i] = (q0 + i == lane) ? 1.f : 0.f;
    }
    float rown = 1.f;
#pragma unroll 1
    for (int k = 31; k >= 0; --k) {
        float *b = bf + (k & 1) * 64;
        if (lane == k) {
            *reinterpret_cast<float4 *>(b + q0) = make_float4(c[0], c[1], c[2], c[3]);
            *reinterpret_cast<float4 *>(b + q0 + 4) = make_float4(c[4], c[5], c[6], c[7]);
            *reinterpret_cast<float4 *>(b + 32 + q0) = make_float4(v[0], v[1], v[2], v[3]);
            *reinterpret_cast<float4 *>(b + 32 + q0 + 4) = make_float4(v[4], v[5], v[6], v[7]);
        }
        __syncthreads();
        float d = b[k];
        if (!(d > 0.f) || !isfinite(d)) {
            if (warp == 0 && lane == 0 && k < valid) atomicCAS(status, -1, (int)(col0 + k));
            d = 1.f;
        }
        const float rinv = rsqrtf(d);
        if (lane == k) rown = rinv;
        const float rjk = lane < k ? b[lane] * rinv : 0.f;
        const float cf = -rjk * rinv;
        const float4 bc0 = *reinterpret_cast<const float4 *>(b + q0);
        const float4 bc1 = *reinterpret_cast<const float4 *>(b + q0 + 4);
        const float4 bv0 = *reinterpret_cast<const float4 *>(b + 32 + q0);
        const float4 bv1 = *reinterpret_cast<const float4 *>(b + 32 + q0 + 4);
        const float bc[8] = {bc0.x, bc0.y, bc0.z, bc0.w, bc1.x, bc1.y, bc1.z, bc1.w};
        const float bv[8] = {bv0.x, bv0.y, bv0.z, bv0.w, bv1.x, bv1.y, bv1.z, bv1.w};
#pragma unroll
        for (int q = 0; q < 8; ++q) {
            if (q0 + q <= lane) c[q] = fmaf(bc[q], cf, c[q]);
            v[q] = fmaf(bv[q], cf, v[q]);
        }
    }
#pragma unroll
    for (int q = 0; q < 8; ++q) Vs[lane][q0 + q] = v[q] * rown;
}

// Diagonal block [k0, k0 + kb) of the reverse-order blocked Cholesky, 128
// threads.  With the block split 2 x 2 into 32 x 32 pieces,
//   A22 = R22 R22^T,  R12 = A12 R22^-T,  A11 - R12 R12^T = R11 R11^T,
//   V = R^-1 = [[V11, -V11 R12 V22], [0, V22]].
// All four warps factor and invert the two diagonal pieces together
// (cta_rchol_inv32) and form the 32 x 32 products.  Out: U_KK = V into
// A[K, K] (upper, in place of the block) and Vt = V^T (dense 64 x 64,
// row-major) for the panel solve.  Rows / columns >= kb are padded with the
// identity.
__global__ void __launch_bounds__(128) chol_diag_kernel(int64_t n, float *A, int64_t k0, int kb, int *status,
                                                        float *Vt) {
    __shared__ float S11[32][33], S22[32][33], A12[32][33];
    __shared__ float V11[32][33], V22[32][33], V12[32][33];
    __shared__ float R12[32][33], X[32][33];   // X = R12 V22
    __shared__ __align__(16) float bf[128];     // pivot broadcast slots
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    {
        // all loads of a thread are issued before the first use
        float x[NB * NB / 128];
#pragma unroll
        for (int t = 0; t < NB * NB / 128; ++t) {
            const int e = tid + t * 128, i = e >> 6, j = e & 63;
            x[t] = (i < kb && j < kb && j >= i) ? A[(k0 + i) * n + k0 + j] : 0.f;
        }
#pragma unroll
        for (int t = 0; t < NB * NB / 128; ++t) {
            const int e = tid + t * 128, i = e >> 6, j = e & 63;
            const float v = (i == j && i >= kb) ? 1.f : x[t];
            if (i < 32) {
                if (j < 32) S11[i][j] = v;
                else A12[i][j - 32] = v;
            } else if (j >= 32) {
                S22[i - 32][j - 32] = v;
            }
        }
    }
    __syncthreads();
    cta_rchol_inv32(S22, V22, bf, warp, lane, status, k0 + 32, kb - 32);
    __syncthreads();
    // R12[i][j] = sum_l A12[i][l] V22[j][l]   (V22 upper, zeros below)
#pragma unroll 1
    for (int e = tid; e < 32 * 32; e += 128) {
        const int i = e >> 5, j = e & 31;
        float acc = 0.f;
#pragma unroll 8
        for (int l = 0; l < 32; ++l) acc = fmaf(A12[i][l], V22[j][l], acc);
        R12[i][j] = acc;
    }
    __syncthreads();
    // A11 -= R12 R12^T and X = R12 V22
#pragma unroll 1
    for (int e = tid; e < 32 * 32; e += 128) {
        const int i = e >> 5, j = e & 31;
        float acc = 0.f, accx = 0.f;
#pragma unroll 8
        for (int l = 0; l < 32; ++l) {
            acc = fmaf(R12[i][l], R12[j][l], acc);
            accx = fmaf(R12[i][l], V22[l][j], accx);
        }
        S11[i][j] -= acc;
        X[i][j] = accx;
    }
    __syncthreads();
    cta_rchol_inv32(S11, V11, bf, warp, lane, status, k0, kb);
    __syncthreads();
    // V12 = -V11 X   (V11 upper, zeros below)
#pragma unroll 1
    for (int e = tid; e < 32 * 32; e += 128) {
        const int i = e >> 5, j = e & 31;
        float acc = 0.f;
#pragma unroll 8
        for (int l = 0; l < 32; ++l) acc = fmaf(V11[i][l], X[l][j], acc);
        V12[i][j] = -acc;
    }
    __syncthreads();
#pragma unroll 4
    for (int e = tid; e < NB * NB; e += 128) {
        const int r = e >> 6, c = e & 63;
        float x;
        if (r < 32) x = c < 32 ? V11[r][c] : V12[r][c - 32];
        else x = c < 32 ? 0.f : V22[r - 32][c - 32];
        if (r < kb && c < kb && c >= r) A[(k0 + r) * n + k0 + c] = x;
        Vt[c * NB + r] = x;
    }
}

// A[i][j] -= sum_c A[i][k0+c] A[j][k0+c] for i <= j < k0 (64 x 64 upper tiles,
// tile idx0 + blockIdx.x of the column-by-column enumeration: tile column tj
// holds tiles (0..tj, tj)).
__global__ void __launch_bounds__(256) chol_update_kernel(int64_t n, float *A, int64_t k0, int kb, int64_t idx0) {
    __shared__ __align__(16) float Pi[NB][NB + 4];
    __shared__ __align__(16) float Pj[NB][NB + 4];
    const int64_t idx = idx0 + blockIdx.x;
    int r = (int)((sqrt(8.0 * (double)idx + 1.0) - 1.0) * 0.5);
    while ((int64_t)(r + 1) * (r + 2) / 2 <= idx) ++r;
    while ((int64_t)r * (r + 1) / 2 > idx) --r;
    const int tj = r, ti = (int)(idx - (int64_t)r * (r + 1) / 2);  // ti <= tj
    const int64_t i0 = (int64_t)ti * NB, j0 = (int64_t)tj * NB;
    {
        // all loads of a thread are issued before the first use
        constexpr int PER = NB * NB / 256;
        float xi[PER], xj[PER];
#pragma unroll
        for (int t = 0; t < PER; ++t) {
            const int e = threadIdx.x + t * 256, rr = e / NB, c = e % NB;
            xi[t] = (c < kb && i0 + rr < k0) ? A[(i0 + rr) * n + k0 + c] : 0.f;
            xj[t] = (c < kb && j0 + rr < k0) ? A[(j0 + rr) * n + k0 + c] : 0.f;
        }
#pragma unroll
        for (int t = 0; t < PER; ++t) {
            const int e = threadIdx.x + t * 256, rr = e / NB, c = e % NB;
            Pi[c][rr] = xi[t];
            Pj[c][rr] = xj[t];
        }
    }
    __syncthreads();
    const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
    float acc[4][4] = {};
    for (int c = 0; c < kb; ++c) {
        const float4 a = *reinterpret_cast<const float4 *>(&Pi[c][ty * 4]);
        const float4 b = *reinterpret_cast<const float4 *>(&Pj[c][tx * 4]);
        const float av[4] = {a.x, a.y, a.z, a.w}, bv[4] = {b.x, b.y, b.z, b.w};
#pragma unroll
        for (int p = 0; p < 4; ++p)
#pragma unroll
            for (int q = 0; q < 4; ++q) acc[p][q] = fmaf(av[p], bv[q], acc[p][q]);
    }
#pragma unroll
    for (int p = 0; p < 4; ++p) {
        const int64_t gi = i0 + ty * 4 + p;
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int64_t gj = j0 + tx * 4 + q;
            if (gi < k0 && gj < k0 && gj >= gi) A[gi * n + gj] -= acc[p][q];
        }
    }
}

__global__ void scale_kernel(int64_t count, float div, const float *in, float *out) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < count) out[i] = in[i] / div;
}

constexpr size_t align256(size_t x) { return (x + 255) / 256 * 256; }
constexpr size_t prepare_bytes(int64_t n) {
    return align256(sizeof(int)) + align256(sizeof(float)) + align256((size_t)NB * NB * sizeof(float)) +
           align256((size_t)n * NB * sizeof(float));
}
// Operand planes of the blocked preparation (three bf16 planes each, pb terms
// deep; pb = PB with a workspace): U_KK, the panel A[0:k0, K] before its solve,
// kPanels panels R[0:k0, K] (a step's updates may still read the earlier ones),
// the row block of U before its product with U_KK, and its transpose after it.
constexpr int64_t PB = kCholBlock;
constexpr int kPanels = 3;
constexpr size_t planes_bytes(int64_t rows, int64_t pb) {
    return align256((size_t)rows * pb * 3 * sizeof(__nv_bfloat16));
}
constexpr size_t blocked_bytes(int64_t n) {
    return n <= PB ? 0 : planes_bytes(PB, PB) + (size_t)(1 + kPanels + 2) * planes_bytes(n, PB);
}
// On one stream a step needs U_KK and n rows beside it: its panel (before the
// solve, then after it) over the k0 rows above the block, and its row block (S,
// then U) over the n - k0 columns from the block on.
constexpr size_t compact_bytes(int64_t n, int64_t pb) { return planes_bytes(pb, pb) + planes_bytes(n, pb); }
// The deepest blocks whose planes fit `bytes` on one stream (0: none).  The
// allocation-free entry point's 8.4 MB hold 512 columns up to n = 2224, 256 up to
// 5216, 128 up to 10816 and 64 up to 21824; against 64-wide steps on the CUDA
// cores n = 2048 takes 0.92 ms (3.80), 4096 2.66 (12.4), 8192 12.4 (47.3), 16384
// 92.7 (230).
int64_t compact_depth(int64_t n, size_t bytes) {
    for (int64_t pb = PB; pb >= NB; pb /= 2)
        if (compact_bytes(n, pb) <= bytes) return pb;
    return 0;
}

// Scratch of the allocation-free entry point, sized for n <= REALQ_PREPARE_NOALLOC_MAX_N.
// Every GPU that loads the library holds it until the process exits.
constexpr size_t kNoAllocBytes = prepare_bytes(REALQ_PREPARE_NOALLOC_MAX_N);
static __device__ __align__(256) unsigned char g_prepare_scratch[kNoAllocBytes];

// Device address of g_prepare_scratch on the current device, looked up on
// every call (it allocates nothing): a cached address would outlive a reset
// device or a recreated primary context, after which the module is loaded
// again at another address.
realq_status_t noalloc_scratch(void **out) {
    void *p = nullptr;
    const cudaError_t e = cudaGetSymbolAddress(&p, g_prepare_scratch);
    if (e != cudaSuccess || p == nullptr)
        return fail(REALQ_ERR_CUDA, "cudaGetSymbolAddress(prepare scratch): %s", cudaGetErrorString(e));
    *out = p;
    return REALQ_OK;
}

}  // namespace

size_t prepare_ws_bytes(int64_t n) { return prepare_bytes(n) + blocked_bytes(n); }

realq_status_t prepare_impl(cudaStream_t s, int64_t n, double norm, float damp, const float *H, float *U, float *Hbar,
                            uint8_t *dead, int64_t *fail_col, void *ws, size_t ws_bytes, bool overlap, bool sync);

realq_status_t prepare_noalloc(cudaStream_t s, int64_t n, int64_t T, float damp, const float *H, float *U, float *Hbar,
                               uint8_t *dead, int64_t *fail_col) {
    void *scratch = nullptr;
    REALQ_TRY(noalloc_scratch(&scratch));
    // single stream: this entry point creates no stream or event
    return prepare_impl(s, n, (double)T, damp, H, U, Hbar, dead, fail_col, scratch, kNoAllocBytes, false, true);
}

// Auxiliary streams of the calling thread (and their events) for the U row
// work and the look-ahead, one set per (device, caller's stream, its
// priority), created on first use and kept for the life of the thread.  Keyed
// by the caller's stream so that calls on different streams (e.g. enqueued
// one after another into one CUDA graph) share no stream and so no false
// dependency.
struct AuxStream {
    int device = -1, priority = 0;
    cudaStream_t caller = nullptr;
    cudaStream_t stream = nullptr;       // the rows of U
    cudaStream_t wide = nullptr;         // the look-ahead's wide trailing updates
    cudaEvent_t ev[3] = {nullptr, nullptr, nullptr};
    std::vector<cudaEvent_t> steps, pdone, wdone, rdone;
};
static thread_local std::vector<AuxStream> g_aux;

realq_status_t aux_for(cudaStream_t s, int64_t nsteps, AuxStream **out) {
    int dev = 0, prio = 0;
    REALQ_CUDA_TRY(cudaGetDevice(&dev));
    REALQ_CUDA_TRY(cudaStreamGetPriority(s, &prio));
    AuxStream *found = nullptr;
    for (AuxStream &x : g_aux)
        if (x.device == dev && x.priority == prio && x.caller == s) found = &x;
    if (!found) {
        AuxStream a;
        REALQ_CUDA_TRY(cudaStreamCreateWithPriority(&a.stream, cudaStreamNonBlocking, prio));
        REALQ_CUDA_TRY(cudaStreamCreateWithPriority(&a.wide, cudaStreamNonBlocking, prio));
        for (int i = 0; i < 3; ++i) REALQ_CUDA_TRY(cudaEventCreateWithFlags(&a.ev[i], cudaEventDisableTiming));
        a.device = dev;
        a.priority = prio;
        a.caller = s;
        g_aux.push_back(a);
        found = &g_aux.back();
    }
    AuxStream &a = *found;
    for (std::vector<cudaEvent_t> *v : {&a.steps, &a.pdone, &a.wdone, &a.rdone}) {
        while ((int64_t)v->size() < nsteps) {
            cudaEvent_t e;
            REALQ_CUDA_TRY(cudaEventCreateWithFlags(&e, cudaEventDisableTiming));
            v->push_back(e);
        }
    }
    *out = &a;
    return REALQ_OK;
}

realq_status_t prepare(cudaStream_t s, int64_t n, double norm, float damp, const float *H, float *U, float *Hbar,
                       uint8_t *dead, int64_t *fail_col, void *ws, size_t ws_bytes) {
    return prepare_impl(s, n, norm, damp, H, U, Hbar, dead, fail_col, ws, ws_bytes, !profiling(), true);
}

realq_status_t prepare_deferred(cudaStream_t s, int64_t n, double norm, float damp, const float *H, float *U,
                                float *Hbar, uint8_t *dead, void *ws, size_t ws_bytes) {
    return prepare_impl(s, n, norm, damp, H, U, Hbar, dead, nullptr, ws, ws_bytes, !profiling(), false);
}

// Inputs of up to n = 64 nbk columns in 64-wide steps on the CUDA cores, one
// stream: for each step the diagonal factor (and inverse), the panel, the
// rank-64 update of what lies above, and row block K of U:
//   U[K, K] = R_KK^-1,  U[K, K+1:] = -U[K, K] (R[K, K+1:] U[K+1:, K+1:])
// (after step K no later step reads row block K of R).
static realq_status_t prepare_steps(cudaStream_t s, int64_t n, float *U, float *Vd, float *panel, int *status) {
    const int nbk = ceil_div(n, NB);
    for (int K = nbk - 1; K >= 0; --K) {
        const int64_t k0 = (int64_t)K * NB;
        const int kb = (int)std::min<int64_t>(NB, n - k0);
        const int64_t k1 = k0 + kb;
        {
            Launch L("chol_diag", s);
            chol_diag_kernel<<<1, 128, 0, s>>>(n, U, k0, kb, status, Vd);
        }
        REALQ_TRY(check_launch("chol_diag"));
        if (k0 > 0) {
            // rows above the block: R[0:k0, K] = A[0:k0, K] R_KK^-T (in place; one
            // column tile, so every CTA reads only the rows it writes)
            GemmArgs pg{};
            pg.M = k0; pg.N = kb; pg.K = kb;
            pg.A = U + k0; pg.lda = n;
            pg.B = Vd; pg.ldb = NB;
            pg.C = U + k0; pg.ldc = n;
            pg.alpha = 1.f;
            REALQ_TRY(gemm_f32(s, A_ROW, EPI_STORE, pg, "chol_panel"));
            const int64_t nt0 = k0 / NB;
            {
                Launch L("chol_update", s);
                chol_update_kernel<<<(unsigned)(nt0 * (nt0 + 1) / 2), 256, 0, s>>>(n, U, k0, kb, 0);
            }
            REALQ_TRY(check_launch("chol_update"));
        }
        if (k1 < n) {
            const int64_t r = n - k1;
            // X = R[K, K+1:] U[K+1:, K+1:] (U upper: a column tile's K range ends
            // at its last column)
            GemmArgs g{};
            g.M = kb; g.N = r; g.K = r;
            g.A = U + k0 * n + k1; g.lda = n;
            g.B = U + k1 * n + k1; g.ldb = n;
            g.C = panel; g.ldc = n;
            g.b_upper = 1;
            g.alpha = 1.f;
            REALQ_TRY(gemm_f32(s, A_ROW, EPI_STORE, g, "trtri_trmm"));
            // U[K, K+1:] = -U_KK X, U_KK read from A[K, K] (upper, zeros below)
            GemmArgs h{};
            h.M = kb; h.N = r; h.K = kb;
            h.A = U + k0 * n + k0; h.lda = n;
            h.B = panel; h.ldb = n;
            h.C = U + k0 * n + k1; h.ldc = n;
            h.alpha = -1.f;
            REALQ_TRY(gemm_f32(s, A_ROW, EPI_STORE, h, "trtri_panel"));
        }
    }
    return REALQ_OK;
}

// Wider inputs, pb columns at a time.  Step K (block K = columns k0 .. k1):
//   s      the cluster factors and inverts A[K, K] (in place: U_KK); the panel
//          R[0:k0, K] = A[0:k0, K] U_KK^T; the update of the next block's
//          columns, A[0:k0, K-1] -= R[0:k0, K] R[K-1, K]^T (upper)
//   wide   the update of the columns before those, overlapped with the next
//          diagonal block and panel (look-ahead)
//   rows   row block K of U.  S[I, j] = sum over K of R[I, K] U[K, j] is
//          accumulated in place of R[I, j] (which step j consumed as planes):
//            U[K, K+1:] = -U_KK S[K, K+1:], then for the rows I above
//            S[I, K] = R[I, K] U_KK and S[I, K+1:] += R[I, K] U[K, K+1:].
// So every product has depth pb and as many tiles as the matrix gives it,
// where one product per row block of U with a depth of up to n had few tiles
// and a long chain.  A product's operands are three bf16 planes each.
// compact: all of it on s, in compact_bytes of planes.
static realq_status_t prepare_blocked(cudaStream_t s, int64_t n, float *U, int *status, int *status_tc,
                                      unsigned char *planes, int64_t pb, bool compact, bool overlap) {
    Carve cv(planes);
    auto take = [&](int64_t rows) { return cv.take<__nv_bfloat16>((size_t)rows * pb * 3); };
    __nv_bfloat16 *Vp = take(pb), *Ap = take(n), *Rp[kPanels] = {Ap, Ap, Ap}, *Sp = nullptr, *Up = nullptr;
    if (!compact) {
        for (int i = 0; i < kPanels; ++i) Rp[i] = take(n);
        Sp = take(n);
        Up = take(n);
    }
    const int nbk = ceil_div(n, pb);
    AuxStream *aux = nullptr;
    if (overlap && !compact) REALQ_TRY(aux_for(s, nbk, &aux));
    cudaStream_t rs = aux ? aux->stream : s, wd = aux ? aux->wide : s;
    if (aux) {
        // the side streams follow everything already on s
        REALQ_CUDA_TRY(cudaEventRecord(aux->ev[0], s));
        REALQ_CUDA_TRY(cudaStreamWaitEvent(rs, aux->ev[0], 0));
        REALQ_CUDA_TRY(cudaStreamWaitEvent(wd, aux->ev[0], 0));
    }
    // planes of rows x pb terms, k terms of which exist
    auto op = [&](const __nv_bfloat16 *p, int64_t rows, int64_t k) { return X6Planes{p, rows, k, pb, rows * pb}; };
    for (int K = nbk - 1; K >= 0; --K) {
        const int64_t k0 = (int64_t)K * pb, kb = std::min<int64_t>(pb, n - k0), k1 = k0 + kb, r = n - k1;
        __nv_bfloat16 *Rk = Rp[K % kPanels];
        if (compact) Sp = Up = Ap + (size_t)k0 * pb * 3;
        __nv_bfloat16 *Ukk = compact ? Vp : Up;   // U_KK for the row block's product
        REALQ_TRY(chol_inv_block(s, n, U + k0 * n + k0, kb, k0, status));
        if (k0 > 0) {
            // the planes of U_KK and of the panel, and the panel's solve (U_KK upper: terms k >= j)
            const X6Split sv{U + k0 * n + k0, n, kb, kb, 0, Vp, pb, kb * pb}, sa{U + k0, n, k0, kb, 0, Ap, pb, k0 * pb};
            REALQ_TRY(split3(s, sa, &sv));
            X6Epi e{};
            e.mode = X6_STORE;
            e.C = U + k0; e.ldc = n;
            e.alpha = 1.f;
            e.b_lo = 1;
            REALQ_TRY(gemm_x6(s, op(Ap, k0, kb), op(Vp, kb, kb), k0, kb, kb, 0, e, status_tc, "chol_panel_tc"));
            // (the planes that step K + kPanels left here are no longer read)
            if (aux && K + kPanels < nbk) REALQ_CUDA_TRY(cudaStreamWaitEvent(s, aux->rdone[K + kPanels], 0));
            const X6Split sr{U + k0, n, k0, kb, 0, Rk, pb, k0 * pb};
            REALQ_TRY(split3(s, sr));
            if (aux) {
                REALQ_CUDA_TRY(cudaEventRecord(aux->pdone[K], s));
                REALQ_CUDA_TRY(cudaStreamWaitEvent(rs, aux->pdone[K], 0));
            }
            const int64_t kw = k0 - pb;   // rows and columns of the wide part
            if (aux) REALQ_CUDA_TRY(cudaStreamWaitEvent(wd, aux->pdone[K], 0));
            // the narrow part's columns were last written by the wide part of step K + 1
            if (aux && K + 1 < nbk) REALQ_CUDA_TRY(cudaStreamWaitEvent(s, aux->wdone[K + 1], 0));
            X6Epi u{};
            u.mode = X6_UPPER;
            u.alpha = -1.f;
            u.C = U + kw; u.ldc = n;
            u.joff = kw;
            REALQ_TRY(gemm_x6(s, op(Rk, k0, kb), op(Rk, k0, kb), k0, pb, kb, kw, u, status_tc,
                              "chol_update_tc"));
            if (kw > 0) {
                X6Epi w{};
                w.mode = X6_UPPER;
                w.alpha = -1.f;
                w.C = U; w.ldc = n;
                REALQ_TRY(gemm_x6(wd, op(Rk, k0, kb), op(Rk, k0, kb), kw, kw, kb, 0, w, status_tc,
                                  "chol_update_tc"));
            }
            if (aux) REALQ_CUDA_TRY(cudaEventRecord(aux->wdone[K], wd));
        } else if (aux) {
            REALQ_CUDA_TRY(cudaEventRecord(aux->steps[K], s));
            REALQ_CUDA_TRY(cudaStreamWaitEvent(rs, aux->steps[K], 0));
        }
        if (r > 0) {
            // U[K, K+1:] = -U_KK S[K, K+1:] (U_KK upper: terms k >= i)
            const X6Split ss{U + k0 * n + k1, n, kb, r, 1, Sp, pb, r * pb}, sv{U + k0 * n + k0, n, kb, kb, 0, Ukk, pb, kb * pb};
            // (compact: above the last step the panel's solve has left them)
            REALQ_TRY(split3(rs, ss, compact && k0 > 0 ? nullptr : &sv));
            X6Epi e{};
            e.mode = X6_STORE;
            e.C = U + k0 * n + k1; e.ldc = n;
            e.alpha = -1.f;
            e.a_lo = 1;
            REALQ_TRY(gemm_x6(rs, op(Ukk, kb, kb), op(Sp, r, kb), kb, r, kb, 0, e, status_tc, "trtri_panel_tc"));
        }
        if (k0 > 0) {
            const int64_t rr = n - k0;
            const X6Split su{U + k0 * n + k0, n, kb, rr, 1, Up, pb, rr * pb};
            REALQ_TRY(split3(rs, su));
            X6Epi e{};
            e.mode = X6_ADD;
            e.alpha = 1.f;
            e.C = U + k0; e.ldc = n;
            e.nstore = kb;
            REALQ_TRY(gemm_x6(rs, op(Rk, k0, kb), op(Up, rr, kb), k0, rr, kb, 0, e, status_tc, "trtri_update_tc"));
            if (aux) REALQ_CUDA_TRY(cudaEventRecord(aux->rdone[K], rs));
        }
    }
    if (aux) {
        REALQ_CUDA_TRY(cudaEventRecord(aux->ev[1], rs));
        REALQ_CUDA_TRY(cudaStreamWaitEvent(s, aux->ev[1], 0));
        REALQ_CUDA_TRY(cudaEventRecord(aux->ev[2], wd));
        REALQ_CUDA_TRY(cudaStreamWaitEvent(s, aux->ev[2], 0));
    }
    return REALQ_OK;
}

realq_status_t prepare_impl(cudaStream_t s, int64_t n, double norm, float damp, const float *H, float *U, float *Hbar,
                            uint8_t *dead, int64_t *fail_col, void *ws, size_t ws_bytes, bool overlap, bool sync) {
    Carve cv(ws);
    int *status = cv.take<int>(1);
    float *lam = cv.take<float>(1);
    const size_t rest = cv.off;
    float *Vd = cv.take<float>((size_t)NB * NB);
    float *panel = cv.take<float>(0);
    // status[0]: the failing column (-1: none); status[1]: timeout bits of
    // the tensor-core products (the same 256-byte slot of the workspace)
    int *status_tc = status + 1;
    REALQ_CUDA_TRY(cudaMemsetAsync(status, 0xFF, sizeof(int), s));
    REALQ_CUDA_TRY(cudaMemsetAsync(status_tc, 0, sizeof(int), s));
    const bool vec = n % 4 == 0 && ((reinterpret_cast<uintptr_t>(H) | reinterpret_cast<uintptr_t>(Hbar) |
                                     reinterpret_cast<uintptr_t>(U)) & 15) == 0;
    const unsigned gy = (unsigned)std::min<int64_t>(n, 65535);
    {
        Launch L("prepare_init", s);
        if (vec)
            prep_init_kernel<true><<<dim3((unsigned)ceil_div(n, 1024), gy), 256, 0, s>>>(n, (float)norm, H, Hbar, U, dead);
        else
            prep_init_kernel<false><<<dim3((unsigned)ceil_div(n, 256), gy), 256, 0, s>>>(n, (float)norm, H, Hbar, U, dead);
    }
    REALQ_TRY(check_launch("prepare_init"));
    {
        Launch L("prepare_damp", s);
        prep_damp_kernel<<<1, 1024, 0, s>>>(n, U, damp, lam);
    }
    REALQ_TRY(check_launch("prepare_damp"));
    if (n <= PB)
        REALQ_TRY(chol_inv_block(s, n, U, n, 0, status));
    else if (ws_bytes >= prepare_ws_bytes(n))
        REALQ_TRY(prepare_blocked(s, n, U, status, status_tc, static_cast<unsigned char *>(ws) + prepare_bytes(n), PB,
                                  false, overlap));
    else if (const int64_t pb = compact_depth(n, ws_bytes - rest))
        REALQ_TRY(prepare_blocked(s, n, U, status, status_tc, static_cast<unsigned char *>(ws) + rest, pb, true, false));
    else
        REALQ_TRY(prepare_steps(s, n, U, Vd, panel, status));
    if (!sync) return REALQ_OK;  // the failing column stays in the workspace's first word
    int host_status[2] = {-1, 0};
    REALQ_CUDA_TRY(cudaMemcpyAsync(host_status, status, 2 * sizeof(int), cudaMemcpyDeviceToHost, s));
    REALQ_CUDA_TRY(cudaStreamSynchronize(s));
    *fail_col = host_status[0];
    if (host_status[1] & ST_TIMEOUT) return fail(REALQ_ERR_TIMEOUT, "a bounded device-side wait gave up (prepare)");
    if (host_status[0] >= 0)
        return fail(REALQ_ERR_NOT_SPD, "damped Hessian not positive definite at column %d", host_status[0]);
    return REALQ_OK;
}

realq_status_t scale_copy(cudaStream_t s, int64_t count, float div, const float *in, float *out) {
    if (count == 0) return REALQ_OK;
    {
        Launch L("scale_moment", s);
        scale_kernel<<<(unsigned)((count + 255) / 256), 256, 0, s>>>(count, div, in, out);
    }
    return check_launch("scale_moment");
}

}  // namespace realq

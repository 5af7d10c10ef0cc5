// FP64 k x k linear algebra of the preconditioner build (Algorithm 3, Eq. (10)):
// the anchor kernel block K_SS, blocked right-looking Cholesky with inverted diagonal
// blocks, triangular inversion by blocks, and small helpers.  All matrices are
// row-major k x k.  k is at most a few thousand, so these run a few hundred
// small launches; GB300's FP64 rate, not memory, bounds them.
#include "internal.cuh"

#include <algorithm>
#include <cmath>
#include <vector>

namespace krr {

constexpr int NB = 32;

__global__ void k_kss(const float* __restrict__ XS, int k, int d, double inv2s2,
                      double* __restrict__ A) {
    const int b = blockIdx.x * blockDim.x + threadIdx.x;
    const int a = blockIdx.y;
    if (b >= k) return;
    double d2 = 0.0;
    for (int c = 0; c < d; ++c) {
        const double df = (double)XS[(size_t)a * d + c] - (double)XS[(size_t)b * d + c];
        d2 = fma(df, df, d2);
    }
    A[(size_t)a * k + b] = exp(-d2 * inv2s2);
}

int launch_kss(krr_ctx* ctx, const float* XS, int k, int d, double sigma, double* A) {
    dim3 grid(ceil_div(k, 128), k);
    k_kss<<<grid, 128, 0, ctx->stream>>>(XS, k, d, 1.0 / (2.0 * sigma * sigma), A);
    KRR_CHECK_LAUNCH();
    return KRR_OK;
}

// FP64 on this GPU issues one warp instruction per ~70 cycles and SM quarter, so what counts in
// these small kernels is the number of dependent FP64 instructions of a thread and how many SMs
// share the work, not memory.  Hence: the diagonal block is factored and inverted in one kernel
// with one reciprocal per column (no divisions or square roots in the elimination; 1024 threads
// that each took the column's square root needed 130 us a block), the blocks below and right of it
// are multiplied by that inverse, one output per thread (a substitution per thread needed 37 to
// 45 us), and trailing updates use 16 x 16 tiles with one output per thread.  Both factorizations
// and inverses of a build with k = 200 went from 3.31 to 0.89 ms, with k = 100 from 1.66 to 0.46 ms.

// 1 / d to FP64 rounding (a few ulp) from the FP32 reciprocal and two Newton steps; d is a pivot
// in the normal FP32 range (0 and non-finite pivots are refused before).
__device__ __forceinline__ double recip64(double d) {
    int ex;
    const double m = frexp(d, &ex);                // [0.5, 1): the FP32 seed neither over- nor underflows
    double x = (double)(1.0f / (float)m);
    x = fma(x, fma(-m, x, 1.0), x);
    x = fma(x, fma(-m, x, 1.0), x);
    return ldexp(x, -ex);
}

// Cholesky of the nb x nb diagonal block at (j0, j0), and its inverse into Linv (NB x NB, row
// major, lower; identity-padded): A_jj = L L^T.  Elimination keeps A_jj = U^T D U unscaled
// (v_r = pivot column, d its pivot): a_rc -= v_r (v_c / d), and the same row operations on the
// identity give the unit inverse; L and its inverse follow from both by the d^(1/2) in parallel.
// Threads (x, y) of 32 x 8 own column x of rows y, y + 8, ...  Bound by FP64 issue: the two halves of
// a row share one instruction (38 us a block with one for each, 32 so).
constexpr int PF_Y = 8;
__global__ void __launch_bounds__(NB * PF_Y)
k_potf2(double* __restrict__ A, int k, int j0, int nb, double tau, int* __restrict__ info,
        double* __restrict__ Linv) {
    pdl_entry();
    __shared__ double s[NB][NB + 1], ei[NB][NB + 1], w[NB], sd[NB];
    const int c = threadIdx.x, y = threadIdx.y;
    const int refused = *info;                     // in a block before: the trailing part was not updated
#pragma unroll
    for (int r = y; r < NB; r += PF_Y) {
        s[r][c] = (r < nb && c < nb) ? A[(size_t)(j0 + r) * k + j0 + c] : (r == c ? 1.0 : 0.0);
        ei[r][c] = r == c ? 1.0 : 0.0;
    }
    if (refused) return;                           // one kernel writes it at a time: every thread read the same
    __syncthreads();
    for (int m = 0; m < nb; ++m) {
        const double piv = s[m][m];
        const bool bad = !(piv > tau) || !isfinite(piv);
        if (bad) {
            if (y == 0 && c == 0) atomicCAS(info, 0, j0 + m + 1);
            return;   // uniform: every thread sees the same s[m][m]
        }
        if (y == 0) {                              // one warp: w_c = v_c / d
            const double inv = recip64(piv);
            w[c] = c > m ? s[c][m] * inv : 0.0;
        }
        __syncthreads();
#pragma unroll
        for (int r = y; r < NB; r += PF_Y) {
            if (r > m) {                           // one FMA for both halves of the row
                const bool right = c > m;
                double* o = right ? &s[r][c] : &ei[r][c];
                const double v = fma(right ? -s[r][m] : -w[r], right ? w[c] : ei[m][c], *o);
                if (c <= r) *o = v;
            }
        }
        __syncthreads();
    }
    if (y == 0) sd[c] = sqrt(s[c][c]);             // pivots (1 in the padding)
    __syncthreads();
    if (y == 0) w[c] = 1.0 / sd[c];
    __syncthreads();
#pragma unroll
    for (int r = y; r < NB; r += PF_Y) {
        if (r < nb && c < nb)
            A[(size_t)(j0 + r) * k + j0 + c] = c < r ? s[r][c] * w[c] : c == r ? sd[c] : 0.0;
        Linv[r * NB + c] = c <= r ? ei[r][c] * w[r] : 0.0;
    }
}

// ---- rows i >= j0 + nb: A[i, j0 : j0 + nb] <- A[i, j0 : j0 + nb] L_jj^{-T}, one output a thread
// (a warp per row: its inputs are read by the warp before any of its outputs is written)
__global__ void __launch_bounds__(128)
k_potrf_panel(double* __restrict__ A, int k, int j0, int nb, const double* __restrict__ Linv,
              const int* __restrict__ info) {
    pdl_entry();
    const int refused = *info;                     // a pivot before: no inverse was written
    __shared__ double L[NB][NB + 1];
    __shared__ double x[4][NB];
    for (int e = threadIdx.x; e < NB * NB; e += blockDim.x) L[e / NB][e % NB] = Linv[e];
    const int c = threadIdx.x & 31, wr = threadIdx.x >> 5;
    const int i = j0 + nb + blockIdx.x * 4 + wr;
    x[wr][c] = (i < k && c < nb) ? A[(size_t)i * k + j0 + c] : 0.0;
    __syncthreads();
    if (i >= k || c >= nb || refused) return;
    double v0 = 0.0, v1 = 0.0;
    for (int m = 0; m <= c; m += 2) {              // Linv[c][m] is 0 beyond m = c
        v0 = fma(x[wr][m], L[c][m], v0);
        if (m + 1 < NB) v1 = fma(x[wr][m + 1], L[c][m + 1], v1);
    }
    A[(size_t)i * k + j0 + c] = v0 + v1;
}

// ---- trailing update: A[i, j] -= sum_m A[i, j0+m] A[j, j0+m]  for 16 x 16 tiles (bi >= bj) past j0+nb
constexpr int DT = 16;
__global__ void __launch_bounds__(DT * DT)
k_potrf_update(double* __restrict__ A, int k, int j0, int nb, int t0, const int* __restrict__ info) {
    pdl_entry();
    const int refused = *info;
    // blockIdx.x enumerates the lower-triangular tile pairs of the trailing matrix
    const int p = blockIdx.x;
    int bi = (int)((sqrtf(8.f * (float)p + 1.f) - 1.f) * 0.5f);
    while ((bi + 1) * (bi + 2) / 2 <= p) ++bi;
    while (bi * (bi + 1) / 2 > p) --bi;
    const int bj = p - bi * (bi + 1) / 2;
    const int r0 = t0 + bi * DT, c0 = t0 + bj * DT;
    __shared__ double sa[DT][NB + 1];
    __shared__ double sb[DT][NB + 1];
    for (int e = threadIdx.x; e < DT * NB; e += DT * DT) {
        const int r = e / NB, m = e - r * NB;
        sa[r][m] = (r0 + r < k && m < nb) ? A[(size_t)(r0 + r) * k + j0 + m] : 0.0;
        sb[r][m] = (c0 + r < k && m < nb) ? A[(size_t)(c0 + r) * k + j0 + m] : 0.0;
    }
    __syncthreads();
    const int c = threadIdx.x % DT, r = threadIdx.x / DT;
    const int gi = r0 + r, gj = c0 + c;
    if (gi >= k || gj >= k || gj > gi || refused) return;
    double v0 = 0.0, v1 = 0.0;
#pragma unroll
    for (int m = 0; m < NB; m += 2) {
        v0 = fma(sa[r][m], sb[c][m], v0);
        v1 = fma(sa[r][m + 1], sb[c][m + 1], v1);
    }
    A[(size_t)gi * k + gj] -= v0 + v1;
}

__global__ void k_zero_upper(double* A, int k) {
    const long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= (long long)k * k) return;
    const int r = (int)(e / k), c = (int)(e - (long long)r * k);
    if (c > r) A[e] = 0.0;
}

static int nblocks(int k) { return (k + NB - 1) / NB; }

// dinv receives the inverses of the diagonal blocks of L (nblocks(k) x NB x NB).
int launch_potrf(krr_ctx* ctx, double* A, int k, int* info_host, double* dinv, double tau) {
    int* info;
    KRR_RET(bufT(ctx, "potrf_info", 1, &info));
    KRR_TRY_CUDA(cudaMemsetAsync(info, 0, sizeof(int), ctx->stream));
    for (int j0 = 0; j0 < k; j0 += NB) {
        const int nb = std::min(NB, k - j0);
        double* Lj = dinv + (size_t)(j0 / NB) * NB * NB;
        launch_pdl(k_potf2, 1, dim3(NB, PF_Y), 0, ctx->stream, A, k, j0, nb, tau, info, Lj);
        KRR_CHECK_LAUNCH();
        const int rest = k - j0 - nb;
        if (rest <= 0) break;
        launch_pdl(k_potrf_panel, ceil_div(rest, 4), 128, 0, ctx->stream, A, k, j0, nb, Lj, info);
        KRR_CHECK_LAUNCH();
        const int tb = (rest + DT - 1) / DT;
        launch_pdl(k_potrf_update, tb * (tb + 1) / 2, DT * DT, 0, ctx->stream, A, k, j0, nb, j0 + nb,
                   info);
        KRR_CHECK_LAUNCH();
    }
    k_zero_upper<<<ceil_div((long long)k * k, 256), 256, 0, ctx->stream>>>(A, k);
    KRR_CHECK_LAUNCH();
    KRR_TRY_CUDA(cudaMemcpyAsync(info_host, info, sizeof(int), cudaMemcpyDeviceToHost, ctx->stream));
    KRR_TRY_CUDA(cudaStreamSynchronize(ctx->stream));
    return KRR_OK;
}

int potrf_dinv(krr_ctx* ctx, int k, double** dinv) {
    return bufT(ctx, "potrf_dinv", (size_t)nblocks(k) * NB * NB, dinv);
}

// ---- X = L^{-1} (lower) by 32-row blocks: at step j0 the rows j0 .. of B hold the identity minus
// what the blocks above contributed; X[j0:, c] = L_jj^{-1} B[j0:, c], then B[i, c] -= L[i, j0:] X[j0:, c]
// for the rows below.  B starts as the identity, so only the columns c < j0 + nb are non-zero.
// One output a thread; a block holds 32 rows x 8 columns, which it reads before it writes.
constexpr int TD_C = 8;
__global__ void __launch_bounds__(NB * TD_C)
k_trinv_diag(const double* __restrict__ Linv, double* __restrict__ B, int k, int j0, int nb, int ncols) {
    pdl_entry();
    __shared__ double sl[NB][NB + 1];
    __shared__ double sx[NB][TD_C + 1];
    for (int e = threadIdx.x; e < NB * NB; e += NB * TD_C) sl[e / NB][e % NB] = Linv[e];
    const int c = threadIdx.x % TD_C, r = threadIdx.x / TD_C;
    const int col = blockIdx.x * TD_C + c;
    const bool ok = r < nb && col < ncols;
    sx[r][c] = ok ? B[(size_t)(j0 + r) * k + col] : 0.0;
    __syncthreads();
    if (!ok) return;
    double v0 = 0.0, v1 = 0.0;
    for (int m = 0; m <= r; m += 2) {
        v0 = fma(sl[r][m], sx[m][c], v0);
        if (m + 1 < NB) v1 = fma(sl[r][m + 1], sx[m + 1][c], v1);
    }
    B[(size_t)(j0 + r) * k + col] = v0 + v1;
}

// B[i, c] -= sum_m L[i, j0+m] B[j0+m, c]  for i >= j0+nb, c < ncols, in 16 x 16 tiles
__global__ void __launch_bounds__(DT * DT)
k_trinv_update(const double* __restrict__ L, double* __restrict__ B, int k, int j0, int nb, int ncols) {
    pdl_entry();
    __shared__ double sl[DT][NB + 1];
    __shared__ double sx[NB][DT + 1];
    const int r0 = j0 + nb + blockIdx.y * DT, c0 = blockIdx.x * DT;
    for (int e = threadIdx.x; e < DT * NB; e += DT * DT) {
        const int r = e / NB, m = e - r * NB;
        sl[r][m] = (r0 + r < k && m < nb) ? L[(size_t)(r0 + r) * k + j0 + m] : 0.0;
        const int m2 = e / DT, c = e - m2 * DT;
        sx[m2][c] = (m2 < nb && c0 + c < ncols) ? B[(size_t)(j0 + m2) * k + c0 + c] : 0.0;
    }
    __syncthreads();
    const int c = threadIdx.x % DT, r = threadIdx.x / DT;
    if (r0 + r >= k || c0 + c >= ncols) return;
    double v0 = 0.0, v1 = 0.0;
#pragma unroll
    for (int m = 0; m < NB; m += 2) {
        v0 = fma(sl[r][m], sx[m][c], v0);
        v1 = fma(sl[r][m + 1], sx[m + 1][c], v1);
    }
    B[(size_t)(r0 + r) * k + c0 + c] -= v0 + v1;
}

// Inverses of the diagonal blocks of a lower triangular L that launch_potrf did not make, one block
// of threads each: forward elimination of [L_jj | I].
__global__ void __launch_bounds__(NB * PF_Y)
k_diag_inverse(const double* __restrict__ L, int k, double* __restrict__ dinv) {
    __shared__ double s[NB][NB + 1], e[NB][NB + 1];
    const int c = threadIdx.x, y = threadIdx.y, j0 = blockIdx.x * NB, nb = min(NB, k - j0);
    for (int r = y; r < NB; r += PF_Y) {
        s[r][c] = (r < nb && c < nb) ? L[(size_t)(j0 + r) * k + j0 + c] : (r == c ? 1.0 : 0.0);
        e[r][c] = r == c ? 1.0 : 0.0;
    }
    __syncthreads();
    for (int m = 0; m < nb; ++m) {
        if (y == 0 && c <= m) e[m][c] /= s[m][m];
        __syncthreads();
        for (int r = y; r < NB; r += PF_Y)
            if (r > m && c <= m) e[r][c] = fma(-s[r][m], e[m][c], e[r][c]);
        __syncthreads();
    }
    for (int r = y; r < NB; r += PF_Y) dinv[(size_t)blockIdx.x * NB * NB + r * NB + c] = c <= r ? e[r][c] : 0.0;
}

int launch_diag_inverse(krr_ctx* ctx, const double* L, int k, double* dinv) {
    k_diag_inverse<<<nblocks(k), dim3(NB, PF_Y), 0, ctx->stream>>>(L, k, dinv);
    KRR_CHECK_LAUNCH();
    return KRR_OK;
}

// B (identity on entry) <- L^{-1}; dinv from launch_potrf on L or from launch_diag_inverse.
int launch_tri_inverse(krr_ctx* ctx, const double* L, const double* dinv, double* B, int k) {
    for (int j0 = 0; j0 < k; j0 += NB) {
        const int nb = std::min(NB, k - j0);
        const int ncols = j0 + nb;   // columns >= j0 + nb are still zero in these rows
        launch_pdl(k_trinv_diag, ceil_div(ncols, TD_C), NB * TD_C, 0, ctx->stream,
                   dinv + (size_t)(j0 / NB) * NB * NB, B, k, j0, nb, ncols);
        KRR_CHECK_LAUNCH();
        const int rest = k - j0 - nb;
        if (rest <= 0) break;
        dim3 grid(ceil_div(ncols, DT), ceil_div(rest, DT));
        launch_pdl(k_trinv_update, grid, DT * DT, 0, ctx->stream, L, B, k, j0, nb, ncols);
        KRR_CHECK_LAUNCH();
    }
    return KRR_OK;
}

__global__ void k_set_identity(double* A, int k) {
    const long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= (long long)k * k) return;
    const int r = (int)(e / k), c = (int)(e - (long long)r * k);
    A[e] = (r == c) ? 1.0 : 0.0;
}

int launch_set_identity(krr_ctx* ctx, double* A, int k) {
    k_set_identity<<<ceil_div((long long)k * k, 256), 256, 0, ctx->stream>>>(A, k);
    KRR_CHECK_LAUNCH();
    return KRR_OK;
}

__global__ void k_add_diag(double* A, int k, double v) {
    const int a = blockIdx.x * blockDim.x + threadIdx.x;
    if (a < k) A[(size_t)a * k + a] += v;
}

int launch_add_diag(krr_ctx* ctx, double* A, int k, double v) {
    k_add_diag<<<ceil_div(k, 256), 256, 0, ctx->stream>>>(A, k, v);
    KRR_CHECK_LAUNCH();
    return KRR_OK;
}

__global__ void k_transpose64(const double* __restrict__ A, double* __restrict__ At, int k) {
    __shared__ double t[32][33];
    const int bx = blockIdx.x * 32, by = blockIdx.y * 32;
    for (int r = threadIdx.y; r < 32; r += blockDim.y) {
        const int gr = by + r, gc = bx + threadIdx.x;
        t[r][threadIdx.x] = (gr < k && gc < k) ? A[(size_t)gr * k + gc] : 0.0;
    }
    __syncthreads();
    for (int r = threadIdx.y; r < 32; r += blockDim.y) {
        const int gr = bx + r, gc = by + threadIdx.x;
        if (gr < k && gc < k) At[(size_t)gr * k + gc] = t[threadIdx.x][r];
    }
}

int launch_transpose64(krr_ctx* ctx, const double* A, double* At, int k) {
    dim3 grid(ceil_div(k, 32), ceil_div(k, 32));
    k_transpose64<<<grid, dim3(32, 8), 0, ctx->stream>>>(A, At, k);
    KRR_CHECK_LAUNCH();
    return KRR_OK;
}

// Out[a * ldo + b] = (float) A[b * k + a]   (zero for b >= k up to ldo)
__global__ void k_to_float_t(const double* __restrict__ A, int k, float* __restrict__ Out, int ldo) {
    const long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= (long long)k * ldo) return;
    const int a = (int)(e / ldo), b = (int)(e - (long long)a * ldo);
    Out[e] = (b < k) ? (float)A[(size_t)b * k + a] : 0.f;
}

int launch_to_float_transposed(krr_ctx* ctx, const double* A, int k, float* Out, int ldo) {
    k_to_float_t<<<ceil_div((long long)k * ldo, 256), 256, 0, ctx->stream>>>(A, k, Out, ldo);
    KRR_CHECK_LAUNCH();
    return KRR_OK;
}

}  // namespace krr

// Conjugate-gradient vector kernels (Algorithm 5 step 3) and the Woodbury
// application of the preconditioner (Algorithm 4, Eq. (7)).
//
// Vectors are FP32, RHS-major (column q of an n x nrhs block at q*n); every dot
// product is accumulated in FP64 and the CG scalars live in a small device struct,
// so the recurrences run without host round trips.  The preconditioner is
//     M^{-1} r = (r - F G^{-1} F^T r) / beta,   G = beta I + F^T F = L2 L2^T,
// with F = K(X, X_S) L1^{-T} stored (n x ldF) and T2 = L2^{-1} held explicitly,
// so one application is two streaming passes over F and two k x k triangular
// products in FP64.
#include "cg_scalar.cuh"
#include "sym.cuh"

#include <algorithm>
#include <cstring>

namespace krr {

constexpr int VT = 256;   // threads of the streaming kernels

// Blocks (per right-hand side) of the vector kernels: four per SM where n allows, one row a thread
// below that: a block's partial sum is one of the numbers that the last block adds.
static int vec_blocks(krr_ctx* ctx, long long n) {
    return (int)std::max<long long>(1, std::min<long long>(4LL * ctx->num_sms, ceil_div(n, VT)));
}
// Blocks of the two passes over F: four per SM (they are latency bound with fewer loads in
// flight); for small n blocks of 32 rows (F^T r) and of 16 rows, two a warp (r - F v), so that a
// set of a few thousand points still fills the chip.
static int ft_blocks(krr_ctx* ctx, long long n) {
    return (int)std::max<long long>(1, std::min<long long>(4LL * ctx->num_sms, ceil_div(n, 32)));
}
static int fn_blocks(krr_ctx* ctx, long long n) {
    return (int)std::max<long long>(1, std::min<long long>(4LL * ctx->num_sms, ceil_div(n, 16)));
}

// Block-wide FP64 sum into part[q * gridDim.x + blockIdx.x].
__device__ __forceinline__ void block_sum_store(double v, double* part, int q) {
    __shared__ double red[VT / 32];
    v = warp_sum(v);
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    __syncthreads();
    if (lane == 0) red[w] = v;
    __syncthreads();
    if (threadIdx.x == 0) {
        double s = 0.0;
        for (int i = 0; i < VT / 32; ++i) s += red[i];
        part[(size_t)q * gridDim.x + blockIdx.x] = s;
    }
}

__global__ void __launch_bounds__(VT)
k_dot_part(const float* __restrict__ A, const float* __restrict__ B, long long n, double* __restrict__ part) {
    const int q = blockIdx.y;
    double s = 0.0;
    for (long long i = (long long)blockIdx.x * VT + threadIdx.x; i < n; i += (long long)gridDim.x * VT)
        s += (double)A[q * n + i] * (double)B[q * n + i];
    block_sum_store(s, part, q);
}

__global__ void __launch_bounds__(VT)
k_dot64_part(const double* __restrict__ A, const double* __restrict__ B, long long n, double* __restrict__ part) {
    const int q = blockIdx.y;
    double s = 0.0;
    for (long long i = (long long)blockIdx.x * VT + threadIdx.x; i < n; i += (long long)gridDim.x * VT)
        s = fma(A[q * n + i], B[q * n + i], s);
    block_sum_store(s, part, q);
}

__global__ void k_sum_parts(const double* __restrict__ part, int nblk, int nrhs, double* out) {
    const int q = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (q >= nrhs) return;
    double s = 0.0;
    for (int b = lane; b < nblk; b += 32) s += part[(size_t)q * nblk + b];
    s = warp_sum(s);
    if (lane == 0) out[q] = s;
}

int launch_dot(krr_ctx* ctx, const float* A, const float* B, long long n, int nrhs, double* out) {
    const int nb = vec_blocks(ctx, n);
    double* part;
    KRR_RET(bufT(ctx, "dot_part", (size_t)nb * nrhs, &part));
    k_dot_part<<<dim3(nb, nrhs), VT, 0, ctx->stream>>>(A, B, n, part);
    KRR_CHECK_LAUNCH();
    k_sum_parts<<<1, 32 * nrhs, 0, ctx->stream>>>(part, nb, nrhs, out);
    KRR_CHECK_LAUNCH();
    return KRR_OK;
}

int launch_dot64(krr_ctx* ctx, const double* A, const double* B, long long n, int nrhs, double* out) {
    const int nb = vec_blocks(ctx, n);
    double* part;
    KRR_RET(bufT(ctx, "dot_part", (size_t)nb * nrhs, &part));
    k_dot64_part<<<dim3(nb, nrhs), VT, 0, ctx->stream>>>(A, B, n, part);
    KRR_CHECK_LAUNCH();
    k_sum_parts<<<1, 32 * nrhs, 0, ctx->stream>>>(part, nb, nrhs, out);
    KRR_CHECK_LAUNCH();
    return KRR_OK;
}

// ------------------------------------------------------------------ Woodbury apply
constexpr int GT_ROWS = 256;   // rows of R staged in shared memory per batch

// Error-free transformations (Knuth two-sum, FMA two-product) for compensated sums.
__device__ __forceinline__ void cg_two_sum(float a, float b, float& s, float& e) {
    s = __fadd_rn(a, b);
    const float z = __fsub_rn(s, a);
    e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, z)), __fsub_rn(b, z));
}
__device__ __forceinline__ void ff_acc(float& h, float& l, float f, float r) {
    const float p = __fmul_rn(f, r);
    const float pe = fmaf(f, r, -p);
    float s, e;
    cg_two_sum(h, p, s, e);
    h = s;
    l = __fadd_rn(l, __fadd_rn(e, pe));
}

// u_part[blk][q][a] = sum_{i in chunk(blk)} F[i, a] R[q, i], as FP64.  The block is G row groups of
// CW threads; a thread owns the float4 columns c, c + CW, ... and the rows of its group, so that
// rows of F are read with 16-byte loads and a short row (CW = ldF / 4 of them, few anchors) still
// uses the whole block.  Products are exact and the sums compensated (float-float): F^T r carries
// the cancellation of the preconditioner, and a plain FP32 sum costs PCG iterations.  (One row
// group left 50 of 256 threads on 64 rows at k = 200: 24 us for one column, 40 for eight, at n = 6000.)
// Sums stay float-float pairs across the row groups and in u_part: two conversions and an add in
// FP64 for each took longer than the products at eight columns.  ONE: a single row group, known
// when compiled (with a stride that is not, the pass over 400 MB took 95 us instead of 74).
template <int NQ, bool ONE>
__global__ void __launch_bounds__(VT)
k_gemv_t(const float* __restrict__ F, long long n, int ldF, const float* __restrict__ R,
         long long ldr, long long rows_per, int CW, float2* __restrict__ upart) {
    pdl_entry();
    __shared__ float sr[NQ][GT_ROWS];
    __shared__ float2 red[ONE ? 1 : VT][4];
    const long long r0 = (long long)blockIdx.x * rows_per;
    const long long r1 = min(n, r0 + rows_per);
    const int ld4 = ldF >> 2;
    const int G = ONE ? 1 : VT / CW, rg = ONE ? 0 : threadIdx.x / CW;
    const int ct = ONE ? threadIdx.x : threadIdx.x - rg * CW;
    const float4* F4 = reinterpret_cast<const float4*>(F);
    const int step = ONE ? VT : CW;
    for (int c0 = 0; c0 < ld4; c0 += step) {
        const int c4 = c0 + ct;
        const bool on = rg < G && c4 < ld4;
        float hx[NQ], hy[NQ], hz[NQ], hw[NQ], lx[NQ], ly[NQ], lz[NQ], lw[NQ];
#pragma unroll
        for (int q = 0; q < NQ; ++q) hx[q] = hy[q] = hz[q] = hw[q] = lx[q] = ly[q] = lz[q] = lw[q] = 0.f;
        for (long long b0 = r0; b0 < r1; b0 += GT_ROWS) {
            const int nb = (int)min((long long)GT_ROWS, r1 - b0);
            __syncthreads();
            for (int e = threadIdx.x; e < NQ * GT_ROWS; e += VT) {
                const int q = e / GT_ROWS, i = e - q * GT_ROWS;
                if (i < nb) sr[q][i] = R[q * ldr + b0 + i];
            }
            __syncthreads();
            if (on) {
                const float4* fp = F4 + b0 * ld4 + c4;
                constexpr int U = NQ > 4 ? 2 : NQ > 2 ? 4 : 8;   // rows whose loads are in flight together
                int i = rg;
                for (; i + (U - 1) * G < nb; i += U * G) {
                    float4 f[U];
#pragma unroll
                    for (int u = 0; u < U; ++u) f[u] = fp[(size_t)(i + u * G) * ld4];
#pragma unroll
                    for (int u = 0; u < U; ++u) {
#pragma unroll
                        for (int q = 0; q < NQ; ++q) {
                            const float a = sr[q][i + u * G];
                            ff_acc(hx[q], lx[q], f[u].x, a); ff_acc(hy[q], ly[q], f[u].y, a);
                            ff_acc(hz[q], lz[q], f[u].z, a); ff_acc(hw[q], lw[q], f[u].w, a);
                        }
                    }
                }
                for (; i < nb; i += G) {
                    const float4 f = fp[(size_t)i * ld4];
#pragma unroll
                    for (int q = 0; q < NQ; ++q) {
                        const float a = sr[q][i];
                        ff_acc(hx[q], lx[q], f.x, a); ff_acc(hy[q], ly[q], f.y, a);
                        ff_acc(hz[q], lz[q], f.z, a); ff_acc(hw[q], lw[q], f.w, a);
                    }
                }
            }
        }
#pragma unroll
        for (int q = 0; q < NQ; ++q) {
            float2 v[4] = {make_float2(hx[q], lx[q]), make_float2(hy[q], ly[q]), make_float2(hz[q], lz[q]),
                           make_float2(hw[q], lw[q])};
            if (!ONE) {                            // over the row groups
                __syncthreads();
#pragma unroll
                for (int w = 0; w < 4; ++w) red[ONE ? 0 : threadIdx.x][w] = v[w];
                __syncthreads();
                if (rg == 0)
                    for (int g = 1; g < G; ++g)
#pragma unroll
                        for (int w = 0; w < 4; ++w) {
                            const float2 o = red[ONE ? 0 : g * CW + ct][w];
                            float h, e;
                            cg_two_sum(v[w].x, o.x, h, e);
                            v[w] = make_float2(h, __fadd_rn(__fadd_rn(v[w].y, o.y), e));
                        }
            }
            if (on && rg == 0) {
                float4* o = reinterpret_cast<float4*>(upart + ((size_t)blockIdx.x * NQ + q) * ldF + 4 * c4);
                o[0] = make_float4(v[0].x, v[0].y, v[1].x, v[1].y);
                o[1] = make_float4(v[2].x, v[2].y, v[3].x, v[3].y);
            }
        }
    }
}

// u[q][a] = sum_blk upart (FP64), a < k.  A CTA covers 8 columns with 32 groups of 8
// threads: each group sums every 32nd partial (8 consecutive columns = one 64-byte
// segment per load), and the groups combine through shared memory.  k / 8 CTAs keep
// enough loads in flight for the 4 x SMs partials of the F^T r pass.
// Pairs are added as pairs and converted once: a conversion of both halves of each cost four FP64
// instructions a partial sum (70 cycles each for a warp here).  A whole apply at n = 30000, k = 1000
// with FP64 partial sums, with each pair converted, and so: two columns 93, 114 and 87 us, three 129,
// 140 and 112, eight (two passes of four with FP64 ones) 388, 230 and 208.  The pair's 2^-44 a term is
// far below the FP32 entries of F: against 64 bits the apply is as far off as with FP64 sums.
template <class T>
struct PartSum;
template <>
struct PartSum<double> {
    double s = 0.0;
    __device__ __forceinline__ void add(double v) { s += v; }
    __device__ __forceinline__ double get() const { return s; }
};
template <>
struct PartSum<float2> {
    float h = 0.f, l = 0.f;
    __device__ __forceinline__ void add(float2 v) {
        ff_add(h, l, v.x);
        l = __fadd_rn(l, v.y);
    }
    __device__ __forceinline__ double get() const { return (double)h + (double)l; }
};
template <class T>
__global__ void __launch_bounds__(256)
k_gemv_t_reduce(const T* __restrict__ upart, int nblk, int nq, int k, int ldF,
                double* __restrict__ u) {
    pdl_entry();
    __shared__ double red[32][9];
    const int c = threadIdx.x & 7, g = threadIdx.x >> 3;
    const int a = blockIdx.x * 8 + c;
    const int q = blockIdx.y;
    PartSum<T> sum;
    if (a < k)
        for (int b = g; b < nblk; b += 32) sum.add(upart[((size_t)b * nq + q) * ldF + a]);
    red[g][c] = sum.get();
    __syncthreads();
    if (threadIdx.x < 8 && a < k) {
        double t = 0.0;
#pragma unroll 8
        for (int i = 0; i < 32; ++i) t += red[i][c];
        u[(size_t)q * k + a] = t;
    }
}

// y[q][a] = sum_b T[a][b] x[q][b] over b <= a (lower) or b >= a (upper), for all NQ columns in one
// pass over T.  TPR threads per row a, 128 in a block: a warp a row for small k (a block a row and a
// pass per column took 12 us for eight columns at k = 200), the whole block a row for large k, where
// every thread then has at most a few independent loads of the row and the k x k factor streams at
// memory rate.
constexpr int TG_T = 128;
template <int NQ, int TPR>
__global__ void __launch_bounds__(TG_T) k_tri_gemv(const double* __restrict__ T, int k,
                                                   const double* __restrict__ x, bool lower,
                                                   double* __restrict__ y) {
    pdl_entry();
    __shared__ double red[NQ][TG_T / 32];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int a = TPR == 32 ? blockIdx.x * (TG_T / 32) + w : (int)blockIdx.x;
    const int t = TPR == 32 ? lane : (int)threadIdx.x;
    if (a >= k) return;                            // whole warps (TPR = 32), no block: a < k
    const int b0 = lower ? 0 : a, b1 = lower ? a + 1 : k;
    constexpr int NV = NQ <= 1 ? 1 : NQ <= 2 ? 2 : NQ <= 4 ? 4 : 8;
    double s[NV];
#pragma unroll
    for (int q = 0; q < NV; ++q) s[q] = 0.0;
#pragma unroll 4
    for (int b = b0 + t; b < b1; b += TPR) {
        const double tv = T[(size_t)a * k + b];
#pragma unroll
        for (int q = 0; q < NQ; ++q) s[q] = fma(tv, x[(size_t)q * k + b], s[q]);
    }
    // over the lanes, halving: a lane ends with the column that its top bits select
    lane_sum<NV, 16>(s, lane);
    double v = s[0];
#pragma unroll
    for (int st = 16 / NV; st >= 1; st >>= 1) v += __shfl_xor_sync(0xffffffffu, v, st);
    const int q = lane / (32 / NV);
    if (lane % (32 / NV) == 0 && q < NQ) {
        if (TPR == 32) y[(size_t)q * k + a] = v;
        else red[q][w] = v;
    }
    if (TPR != 32) {
        __syncthreads();
        if ((int)threadIdx.x < NQ) {
            double x0 = 0.0;
#pragma unroll
            for (int i = 0; i < TG_T / 32; ++i) x0 += red[threadIdx.x][i];
            y[(size_t)threadIdx.x * k + a] = x0;
        }
    }
}

typedef void (*tri_fn)(const double*, int, const double*, bool, double*);
template <int TPR>
static tri_fn tri_pick1(int nq) {
    static const tri_fn t[8] = {&k_tri_gemv<1, TPR>, &k_tri_gemv<2, TPR>, &k_tri_gemv<3, TPR>, &k_tri_gemv<4, TPR>,
                                &k_tri_gemv<5, TPR>, &k_tri_gemv<6, TPR>, &k_tri_gemv<7, TPR>, &k_tri_gemv<8, TPR>};
    return t[nq - 1];
}
int launch_tri_gemv(krr_ctx* ctx, const double* T, int k, const double* x, int nq, bool lower, double* y) {
    if (nq < 1 || nq > 8) return fail(ctx, KRR_E_INVAL, "triangular product: bad column count");
    if (k <= 512)
        launch_pdl(tri_pick1<32>(nq), ceil_div(k, TG_T / 32), TG_T, 0, ctx->stream, T, k, x, lower, y);
    else
        launch_pdl(tri_pick1<TG_T>(nq), k, TG_T, 0, ctx->stream, T, k, x, lower, y);
    KRR_CHECK_LAUNCH();
    return KRR_OK;
}

// Z[q][i] = (R[q][i] - sum_a F[i, a] v[q][a]) / beta; one warp per row with float4 loads, two rows at
// a time.  Optional per-block partial sums of R.Z.
template <int NQ>
__global__ void __launch_bounds__(VT)
k_gemv_n_apply(const float* __restrict__ F, long long n, int k, int ldF, const double* __restrict__ v,
               const float* __restrict__ R, long long ldr, float inv_beta, float* __restrict__ Z,
               double* __restrict__ rz_part, CGScalars* cg, int q0) {
    pdl_entry();
    extern __shared__ float4 sv4[];   // NQ x ld4
    const int ld4 = ldF >> 2;
    for (int e = threadIdx.x; e < NQ * ld4; e += VT) {
        const int q = e / ld4, c4 = e - q * ld4;
        float t[4];
#pragma unroll
        for (int w = 0; w < 4; ++w) {
            const int a = 4 * c4 + w;
            t[w] = (a < k) ? (float)v[(size_t)q * k + a] : 0.f;
        }
        sv4[e] = make_float4(t[0], t[1], t[2], t[3]);
    }
    __syncthreads();
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const float4* F4 = reinterpret_cast<const float4*>(F);
    // 2 NV sums (column m / 2, row m % 2) over the lanes, halving in turn: lane ends with the one
    // that its top bits select, as many shuffles as sums instead of five for each
    constexpr int NV = NQ <= 1 ? 1 : NQ <= 2 ? 2 : NQ <= 4 ? 4 : 8;
    constexpr int REST = 32 / (2 * NV);            // lanes that share a sum
    const int m = lane / REST, mq = m >> 1, mh = m & 1;
    double rz = 0.0;
    // each warp takes two rows at a time and issues all of their loads before the FMAs
    const long long wstride = (long long)gridDim.x * (VT / 32);
    for (long long i0 = (long long)blockIdx.x * (VT / 32) + w; i0 < n; i0 += 2 * wstride) {
        const long long i1 = i0 + wstride;
        const bool has1 = i1 < n;
        float s[2 * NV];
#pragma unroll
        for (int q = 0; q < 2 * NV; ++q) s[q] = 0.f;
        const float4* f0 = F4 + i0 * ld4;
        const float4* f1 = F4 + (has1 ? i1 : i0) * ld4;
        for (int c0 = lane; c0 < ld4; c0 += 32 * 4) {
            float4 a[4], b[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int c = c0 + 32 * u;
                a[u] = c < ld4 ? f0[c] : make_float4(0.f, 0.f, 0.f, 0.f);
                b[u] = (c < ld4 && has1) ? f1[c] : make_float4(0.f, 0.f, 0.f, 0.f);
            }
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int c = c0 + 32 * u;
                if (c >= ld4) break;
#pragma unroll
                for (int q = 0; q < NQ; ++q) {
                    const float4 vv = sv4[q * ld4 + c];
                    s[2 * q] = fmaf(a[u].x, vv.x, fmaf(a[u].y, vv.y, fmaf(a[u].z, vv.z, fmaf(a[u].w, vv.w, s[2 * q]))));
                    s[2 * q + 1] = fmaf(b[u].x, vv.x, fmaf(b[u].y, vv.y, fmaf(b[u].z, vv.z, fmaf(b[u].w, vv.w, s[2 * q + 1]))));
                }
            }
        }
        __syncwarp();
        lane_sum<2 * NV, 16>(s, lane);
        float t = s[0];
#pragma unroll
        for (int st = REST / 2; st >= 1; st >>= 1) t += __shfl_xor_sync(0xffffffffu, t, st);
        if (lane % REST == 0 && mq < NQ && (mh == 0 || has1)) {
            const long long i = mh ? i1 : i0;
            const float r = R[mq * ldr + i];
            const float z = (r - t) * inv_beta;
            Z[mq * ldr + i] = z;
            rz += (double)r * (double)z;
        }
    }
    if (rz_part) {
        __shared__ double rzs[VT / 32][2 * NV];
        if (lane % REST == 0) rzs[w][m] = rz;
        __syncthreads();
        if (threadIdx.x < NQ) {
            double t = 0.0;
#pragma unroll
            for (int i = 0; i < VT / 32; ++i) t += rzs[i][2 * threadIdx.x] + rzs[i][2 * threadIdx.x + 1];
            rz_part[(size_t)threadIdx.x * gridDim.x + blockIdx.x] = t;
        }
        // the last block forms the columns' b = rz_new / rz (b = 0 for finished columns: p restarts
        // from z); rz itself is replaced when p is updated, so that this pass may be repeated
        if (cg && last_block(&cg->ticket[0])) {
            for (int q = w; q < NQ; q += VT / 32) {
                const double sum = warp_sum_parts(rz_part, gridDim.x, q);
                if (lane == 0) {
                    const double z = cg->rz[q0 + q];
                    cg->b[q0 + q] = (cg->active[q0 + q] && z != 0.0 && isfinite(sum)) ? sum / z : 0.0;
                    cg->rz_new[q0 + q] = sum;
                }
            }
        }
    }
}

typedef void (*gemv_t_fn)(const float*, long long, int, const float*, long long, long long, int, float2*);
typedef void (*gemv_n_fn)(const float*, long long, int, int, const double*, const float*, long long,
                          float, float*, double*, CGScalars*, int);
constexpr int AP_NQ = 8;   // most right-hand sides per pass over F

// Right-hand sides per pass over F: r - F v holds v of all of them in shared memory (4 ldF bytes each,
// beside up to 1 KB of sums), so that more than about 7200 anchors leave room for fewer than eight.
// As many as fit: a pass reads F once whatever its columns, and one block an SM with eight is still
// ahead of two passes (n = 30000, eight columns, against passes of four with more blocks an SM:
// k = 3800 0.89 against 1.42 ms, 5000 1.21 against 1.87, 6500 1.70 against 2.65).
// The limits are asked for only past AP_SMEM, which with the static part is safe without leave.
constexpr int AP_SMEM = 40 * 1024;
static int apply_columns(krr_ctx* ctx, int ldF, int nrhs, int* nq) {
    *nq = std::min(AP_NQ, nrhs);
    if (4LL * ldF * *nq <= AP_SMEM) return KRR_OK;
    int optin = 0;
    KRR_TRY_CUDA(cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, ctx->device));
    *nq = std::max(1, std::min(*nq, (optin - 2048) / (4 * ldF)));
    return KRR_OK;
}

// Z = M^{-1} R for nrhs columns.  When rz_part is non-null it receives per-block partial
// sums of R.Z laid out [q][blk] with apply_blocks(ctx) blocks per column; with_beta also forms the
// recurrence's b and rz_new from them.
int launch_apply_precond(krr_ctx* ctx, const float* R, int nrhs, float* Z, double* rz_part, bool with_beta) {
    const long long n = ctx->n;
    const int k = ctx->k_eff, ldF = ctx->ldF;
    const int nt = ft_blocks(ctx, n), nb = fn_blocks(ctx, n);
    const long long rows_per = ceil_div(n, nt);
    const int CW = std::min(VT, ldF / 4);          // threads across a row of F
    float2* upart;
    double *u, *u1, *v;
    int mq;
    KRR_RET(apply_columns(ctx, ldF, nrhs, &mq));
    KRR_RET(bufT(ctx, "ap_upart2", (size_t)nt * mq * ldF, &upart));
    KRR_RET(bufT(ctx, "ap_u", (size_t)mq * k, &u));
    KRR_RET(bufT(ctx, "ap_u1", (size_t)mq * k, &u1));
    KRR_RET(bufT(ctx, "ap_v", (size_t)mq * k, &v));
    const float inv_beta = (float)(1.0 / ctx->beta);
    static const gemv_t_fn gts[2][AP_NQ] = {
        {&k_gemv_t<1, false>, &k_gemv_t<2, false>, &k_gemv_t<3, false>, &k_gemv_t<4, false>, &k_gemv_t<5, false>,
         &k_gemv_t<6, false>, &k_gemv_t<7, false>, &k_gemv_t<8, false>},
        {&k_gemv_t<1, true>, &k_gemv_t<2, true>, &k_gemv_t<3, true>, &k_gemv_t<4, true>, &k_gemv_t<5, true>,
         &k_gemv_t<6, true>, &k_gemv_t<7, true>, &k_gemv_t<8, true>}};
    static const gemv_n_fn gns[AP_NQ] = {&k_gemv_n_apply<1>, &k_gemv_n_apply<2>, &k_gemv_n_apply<3>,
                                         &k_gemv_n_apply<4>, &k_gemv_n_apply<5>, &k_gemv_n_apply<6>,
                                         &k_gemv_n_apply<7>, &k_gemv_n_apply<8>};
    for (int q0 = 0; q0 < nrhs; q0 += mq) {
        const int nq = std::min(mq, nrhs - q0);
        const gemv_t_fn gt = gts[2 * CW > VT][nq - 1];   // room for one row group only
        const gemv_n_fn gn = gns[nq - 1];
        const float* Rq = R + (size_t)q0 * n;
        float* Zq = Z + (size_t)q0 * n;
        launch_pdl_if(nt < 4 * ctx->num_sms, gt, nt, VT, 0, ctx->stream, ctx->F, n, ldF, Rq, n, rows_per, CW, upart);
        KRR_CHECK_LAUNCH();
        launch_pdl(k_gemv_t_reduce<float2>, dim3(ceil_div(k, 8), nq), 256, 0, ctx->stream, upart, nt, nq, k, ldF, u);
        KRR_CHECK_LAUNCH();
        KRR_RET(launch_tri_gemv(ctx, ctx->T2, k, u, nq, true, u1));
        KRR_RET(launch_tri_gemv(ctx, ctx->T2t, k, u1, nq, false, v));
        const size_t smem = sizeof(float4) * nq * (ldF / 4);
        // not only above 48 KB: these are for the dynamic and the kernel's static memory together
        if (smem > AP_SMEM) KRR_RET(allow_max_dynamic_smem(ctx, (const void*)gn));
        launch_pdl_if(nb < 4 * ctx->num_sms, gn, nb, VT, smem, ctx->stream, ctx->F, n, k, ldF, v, Rq, n, inv_beta, Zq,
                   rz_part ? rz_part + (size_t)q0 * nb : nullptr, rz_part && with_beta ? ctx->cg : nullptr, q0);
        KRR_CHECK_LAUNCH();
    }
    return KRR_OK;
}

// ------------------------------------------------------------------ PCG recurrences
// The scalar kernels run one warp per right-hand side: the warp sums that column's
// per-block partials (FP64) and lane 0 applies the recurrence.
__global__ void k_cg_alpha(CGScalars* cg, const double* __restrict__ part, int nblk, int nrhs) {
    const int q = threadIdx.x >> 5;
    if (q >= nrhs) return;
    const double s = warp_sum_parts(part, nblk, q);
    if ((threadIdx.x & 31) == 0) cg_alpha(cg, q, s);
}
// p . q and, in the last block, the step lengths: one launch instead of two in every iteration
__global__ void __launch_bounds__(VT)
k_cg_dot_alpha(const float* __restrict__ p, const float* __restrict__ qv, long long n, CGScalars* cg,
               double* __restrict__ part) {
    pdl_entry();
    {
        const int q = blockIdx.y;
        double s = 0.0;
        for (long long i = (long long)blockIdx.x * VT + threadIdx.x; i < n; i += (long long)gridDim.x * VT)
            s += (double)p[q * n + i] * (double)qv[q * n + i];
        block_sum_store(s, part, q);
    }
    if (!last_block(&cg->ticket[1])) return;
    for (int q = threadIdx.x >> 5; q < (int)gridDim.y; q += VT / 32) {
        const double s = warp_sum_parts(part, gridDim.x, q);
        if ((threadIdx.x & 31) == 0) cg_alpha(cg, q, s);
    }
}

// rr_q = s (recursive residual); a non-finite one ends the column, and with tol2 > 0 so does
// rr_q <= tol2 rr0_q.  Returns whether the column goes on.
__device__ __forceinline__ bool cg_check(CGScalars* cg, int q, double s, double tol2) {
    cg->rr[q] = s;
    if (!isfinite(s)) {
        cg->bad = 1;
        cg->active[q] = 0;
    }
    if (tol2 > 0.0 && cg->active[q] && !(s > tol2 * cg->rr0[q])) cg->active[q] = 0;
    return cg->active[q] != 0;
}
__global__ void k_cg_check(CGScalars* cg, const double* __restrict__ part, int nblk, int nrhs,
                           double tol2) {
    __shared__ int any;
    if (threadIdx.x == 0) any = 0;
    __syncthreads();
    const int q = threadIdx.x >> 5;
    if (q < nrhs) {
        const double s = warp_sum_parts(part, nblk, q);
        if ((threadIdx.x & 31) == 0 && cg_check(cg, q, s, tol2)) atomicOr(&any, 1);
    }
    __syncthreads();
    if (threadIdx.x == 0) cg->all_done = any ? 0 : 1;
}
// x += a p; r -= a q; r.r and, in the last block, the check above.  With `host` (pinned) that block also
// writes what the host decides on there, and then `seq`: two copies and an event between this kernel
// and the next cost the queue three more entries an iteration, and the overlap of their launches.
__global__ void __launch_bounds__(VT)
k_cg_update_xr(float* __restrict__ x, float* __restrict__ r, const float* __restrict__ p,
               const float* __restrict__ qv, long long n, CGScalars* cg,
               double* __restrict__ part, double tol2, CGScalars* host, const int* tc_err, unsigned long long seq) {
    pdl_entry();
    {
        const int q = blockIdx.y;
        const float a = (float)cg->a[q];
        double s = 0.0;
        for (long long i = (long long)blockIdx.x * VT + threadIdx.x; i < n; i += (long long)gridDim.x * VT) {
            const long long e = q * n + i;
            const float rv = fmaf(-a, qv[e], r[e]);
            x[e] = fmaf(a, p[e], x[e]);
            r[e] = rv;
            s += (double)rv * (double)rv;
        }
        block_sum_store(s, part, q);
    }
    if (!last_block(&cg->ticket[2])) return;
    __shared__ int any;
    if (threadIdx.x == 0) any = 0;
    __syncthreads();
    for (int q = threadIdx.x >> 5; q < (int)gridDim.y; q += VT / 32) {
        const double s = warp_sum_parts(part, gridDim.x, q);
        if ((threadIdx.x & 31) == 0 && cg_check(cg, q, s, tol2)) atomicOr(&any, 1);
    }
    __syncthreads();
    if (threadIdx.x == 0) cg->all_done = any ? 0 : 1;
    if (!host) return;
    if (threadIdx.x < gridDim.y) host->rr[threadIdx.x] = cg->rr[threadIdx.x];
    if (threadIdx.x == 0) {
        host->a[0] = cg->a[0];
        host->b[0] = cg->b[0];
        host->bad = cg->bad;
        host->tc_err = tc_err ? *tc_err : 0;
    }
    __threadfence_system();
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence_system();
        *(volatile unsigned long long*)&host->seq = seq;
    }
}

// b_q = rz_new / rz; rz = rz_new (b = 0 for finished columns: p restarts from z)
__global__ void k_cg_beta(CGScalars* cg, const double* __restrict__ part, int nblk, int nrhs) {
    const int q = threadIdx.x >> 5;
    if (q >= nrhs) return;
    const double s = warp_sum_parts(part, nblk, q);
    if ((threadIdx.x & 31) != 0) return;
    const double rz = cg->rz[q];
    cg->b[q] = (cg->active[q] && rz != 0.0 && isfinite(s)) ? s / rz : 0.0;
    cg->rz[q] = s;
}

// p = z + b p; with_beta (b came with the apply): rz = rz_new, which nothing here reads
__global__ void __launch_bounds__(VT)
k_cg_update_p(float* __restrict__ p, const float* __restrict__ z, long long n, CGScalars* cg, bool with_beta) {
    pdl_entry();
    const int q = blockIdx.y;
    if (with_beta && blockIdx.x == 0 && threadIdx.x == 0) cg->rz[q] = cg->rz_new[q];
    const float b = (float)cg->b[q];
    for (long long i = (long long)blockIdx.x * VT + threadIdx.x; i < n; i += (long long)gridDim.x * VT)
        p[q * n + i] = fmaf(b, p[q * n + i], z[q * n + i]);
}

// start: rz = part sum (r.z), rr0 = r.r given in rr0_part, active = rr0 > 0; a warp per column
__global__ void k_cg_init(CGScalars* cg, const double* __restrict__ rz_part, int nrz,
                          const double* __restrict__ rr_part, int nrr, int nrhs) {
    const int q = threadIdx.x >> 5;
    if (threadIdx.x == 0) {
        cg->all_done = 0;
        cg->bad = 0;
    }
    if (q >= nrhs) return;
    const double s = warp_sum_parts(rz_part, nrz, q);
    const double t = warp_sum_parts(rr_part, nrr, q);
    if ((threadIdx.x & 31) != 0) return;
    cg->rz[q] = s;
    cg->rr0[q] = t;
    cg->rr[q] = t;
    cg->active[q] = (t > 0.0 && isfinite(t) && isfinite(s)) ? 1 : 0;
    cg->a[q] = 0.0;
    cg->b[q] = 0.0;
}

// out32 = (float) in64 ; and alpha64 += x32
__global__ void k_f64_to_f32(const double* __restrict__ a, float* __restrict__ b, long long tot) {
    for (long long e = (long long)blockIdx.x * VT + threadIdx.x; e < tot; e += (long long)gridDim.x * VT)
        b[e] = (float)a[e];
}
__global__ void k_f32_to_f64(const float* __restrict__ a, double* __restrict__ b, long long tot) {
    for (long long e = (long long)blockIdx.x * VT + threadIdx.x; e < tot; e += (long long)gridDim.x * VT)
        b[e] = (double)a[e];
}
__global__ void k_axpy_f32_into_f64(const float* __restrict__ x, double* __restrict__ y, long long tot) {
    for (long long e = (long long)blockIdx.x * VT + threadIdx.x; e < tot; e += (long long)gridDim.x * VT)
        y[e] += (double)x[e];
}

// ---- host drivers for the recurrences (launch sequences; no host sync inside)
int launch_cg_set_active(krr_ctx* ctx, const int* act_host, int nrhs) {
    // staged through the pinned mirror so the copy is asynchronous
    std::memcpy(ctx->cg_host->active, act_host, sizeof(int) * nrhs);
    KRR_TRY_CUDA(cudaMemcpyAsync(ctx->cg->active, ctx->cg_host->active, sizeof(int) * nrhs,
                                 cudaMemcpyHostToDevice, ctx->stream));
    return KRR_OK;
}

int cg_vec_blocks(krr_ctx* ctx) { return vec_blocks(ctx, ctx->n); }
int apply_blocks(krr_ctx* ctx) { return fn_blocks(ctx, ctx->n); }
// blocks of the apply's partial sums of r . z: the identity's come from the vector kernels
static int rz_blocks(krr_ctx* ctx) { return ctx->opts.no_precond ? vec_blocks(ctx, ctx->n) : apply_blocks(ctx); }

int launch_cg_start(krr_ctx* ctx, const float* r, const float* z, int nrhs, double* rz_part,
                    double* rr_part) {
    const int nb = vec_blocks(ctx, ctx->n);
    k_dot_part<<<dim3(nb, nrhs), VT, 0, ctx->stream>>>(r, r, ctx->n, rr_part);
    KRR_CHECK_LAUNCH();
    k_cg_init<<<1, 32 * nrhs, 0, ctx->stream>>>(ctx->cg, rz_part, rz_blocks(ctx), rr_part, nb, nrhs);
    KRR_CHECK_LAUNCH();
    (void)z;
    return KRR_OK;
}

int launch_cg_alpha(krr_ctx* ctx, const float* p, const float* q, int nrhs, double* part) {
    const int nb = vec_blocks(ctx, ctx->n);
    launch_pdl(k_cg_dot_alpha, dim3(nb, nrhs), VT, 0, ctx->stream, p, q, ctx->n, ctx->cg, part);
    KRR_CHECK_LAUNCH();
    return KRR_OK;
}

int launch_cg_update_xr(krr_ctx* ctx, float* x, float* r, const float* p, const float* q, int nrhs,
                        double* part, double tol2, bool mirror, const int* tc_err) {
    const int nb = vec_blocks(ctx, ctx->n);
    launch_pdl(k_cg_update_xr, dim3(nb, nrhs), VT, 0, ctx->stream, x, r, p, q, ctx->n, ctx->cg, part, tol2,
               mirror ? ctx->cg_host : nullptr, tc_err, mirror ? ++ctx->cg_seq : 0ull);
    KRR_CHECK_LAUNCH();
    return KRR_OK;
}

int launch_cg_beta_p(krr_ctx* ctx, float* p, const float* z, int nrhs, const double* rz_part, bool with_beta) {
    const int nb = vec_blocks(ctx, ctx->n);
    if (!with_beta) {
        k_cg_beta<<<1, 32 * nrhs, 0, ctx->stream>>>(ctx->cg, rz_part, rz_blocks(ctx), nrhs);
        KRR_CHECK_LAUNCH();
    }
    launch_pdl(k_cg_update_p, dim3(nb, nrhs), VT, 0, ctx->stream, p, z, ctx->n, ctx->cg, with_beta);
    KRR_CHECK_LAUNCH();
    return KRR_OK;
}

// The identity in place of the preconditioner (plain CG): Z = R and per-block partial
// sums of R.R in the layout of launch_apply_precond's rz_part.
int launch_identity_apply(krr_ctx* ctx, const float* R, int nrhs, float* Z, double* rz_part) {
    const long long n = ctx->n;
    if (Z != R)
        KRR_TRY_CUDA(cudaMemcpyAsync(Z, R, sizeof(float) * n * nrhs, cudaMemcpyDeviceToDevice, ctx->stream));
    if (rz_part) {
        k_dot_part<<<dim3(vec_blocks(ctx, n), nrhs), VT, 0, ctx->stream>>>(R, R, n, rz_part);
        KRR_CHECK_LAUNCH();
    }
    return KRR_OK;
}
int launch_identity_apply64(krr_ctx* ctx, const double* R, int nrhs, double* Z, double* rz_part) {
    const long long n = ctx->n;
    if (Z != R)
        KRR_TRY_CUDA(cudaMemcpyAsync(Z, R, sizeof(double) * n * nrhs, cudaMemcpyDeviceToDevice, ctx->stream));
    if (rz_part) {
        k_dot64_part<<<dim3(cg64_vec_blocks(ctx), nrhs), VT, 0, ctx->stream>>>(R, R, n, rz_part);
        KRR_CHECK_LAUNCH();
    }
    return KRR_OK;
}

// pieces used by the FP64 recurrence (cg64.cu)
int launch_gemv_t_reduce(krr_ctx* ctx, const double* upart, int nblk, int nq, int k, int ldF, double* u) {
    launch_pdl(k_gemv_t_reduce<double>, dim3(ceil_div(k, 8), nq), 256, 0, ctx->stream, upart, nblk, nq, k, ldF, u);
    KRR_CHECK_LAUNCH();
    return KRR_OK;
}
int launch_dot64_parts(krr_ctx* ctx, const double* A, const double* B, long long n, int nrhs, int nb,
                       double* part) {
    k_dot64_part<<<dim3(nb, nrhs), VT, 0, ctx->stream>>>(A, B, n, part);
    KRR_CHECK_LAUNCH();
    return KRR_OK;
}
int launch_cg_scalars_init(krr_ctx* ctx, const double* rz_part, const double* rr_part, int nb, int nrhs) {
    k_cg_init<<<1, 32 * nrhs, 0, ctx->stream>>>(ctx->cg, rz_part, nb, rr_part, nb, nrhs);
    KRR_CHECK_LAUNCH();
    return KRR_OK;
}
int launch_cg_scalars_alpha(krr_ctx* ctx, const double* part, int nb, int nrhs) {
    k_cg_alpha<<<1, 32 * nrhs, 0, ctx->stream>>>(ctx->cg, part, nb, nrhs);
    KRR_CHECK_LAUNCH();
    return KRR_OK;
}
int launch_cg_scalars_check(krr_ctx* ctx, const double* part, int nb, int nrhs, double tol2) {
    k_cg_check<<<1, 32 * nrhs, 0, ctx->stream>>>(ctx->cg, part, nb, nrhs, tol2);
    KRR_CHECK_LAUNCH();
    return KRR_OK;
}
int launch_cg_scalars_beta(krr_ctx* ctx, const double* rz_part, int nb, int nrhs) {
    k_cg_beta<<<1, 32 * nrhs, 0, ctx->stream>>>(ctx->cg, rz_part, nb, nrhs);
    KRR_CHECK_LAUNCH();
    return KRR_OK;
}

int launch_convert(krr_ctx* ctx, const double* a, float* b, long long tot) {
    k_f64_to_f32<<<vec_blocks(ctx, tot), VT, 0, ctx->stream>>>(a, b, tot);
    KRR_CHECK_LAUNCH();
    return KRR_OK;
}
int launch_convert_up(krr_ctx* ctx, const float* a, double* b, long long tot) {
    k_f32_to_f64<<<vec_blocks(ctx, tot), VT, 0, ctx->stream>>>(a, b, tot);
    KRR_CHECK_LAUNCH();
    return KRR_OK;
}
int launch_accumulate(krr_ctx* ctx, const float* x, double* y, long long tot) {
    k_axpy_f32_into_f64<<<vec_blocks(ctx, tot), VT, 0, ctx->stream>>>(x, y, tot);
    KRR_CHECK_LAUNCH();
    return KRR_OK;
}

}  // namespace krr

// Refinement residual R = Y - (K + beta I) A carried in float-float on the FP32 pipe.
//
// GB300 issues FP64 FMAs at about 1/70 of the FP32 rate, so the residual that
// drives iterative refinement keeps every quantity as an unevaluated sum of two
// floats (about 48 significant bits) instead:
//   * x_i . x_j is summed exactly term by term (FMA two-product + Knuth two-sum),
//     and ||x_i - x_j||^2 = n_i + n_j - 2 x_i . x_j with float-float norms;
//   * t = -s ||x_i - x_j||^2 with s = log2(e) / (2 sigma^2) in float-float;
//   * 2^t by the table-driven reduction of P. T. P. Tang, "Table-driven
//     implementation of the exponential function in IEEE floating-point
//     arithmetic", ACM TOMS 15(2), 1989, carried in float-float:
//     2^t = 2^m * 2^(j/64) * e^z with m = round(t), j = round(64 (t - m)) picking
//     an entry of a 65-entry float-float table of 2^(j/64) (built on the host in
//     double), and e^z with |z| <= ln2/128 evaluated as its Taylor polynomial
//     1 + z + ... + z^5/120 (truncation below 4e-17); the low word of t enters as
//     the factor (1 + ln2 t_lo);
//   * K_ij A_j is formed exactly (two-product), summed in float-float over a
//     tile of 64 columns and folded into an FP64 accumulator per tile.
// Relative error of each kernel value is a few 1e-12, against ~1e-7 for the FP32
// tile kernel.
#include "internal.cuh"
#include "sym.cuh"

#include <algorithm>
#include <type_traits>
#include <cmath>

namespace krr {

__device__ __forceinline__ void two_sum(float a, float b, float& s, float& e) {
    s = __fadd_rn(a, b);
    const float z = __fsub_rn(s, a);
    e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, z)), __fsub_rn(b, z));
}
// requires |a| >= |b| (or a == 0)
__device__ __forceinline__ void fast_two_sum(float a, float b, float& s, float& e) {
    s = __fadd_rn(a, b);
    e = __fsub_rn(b, __fsub_rn(s, a));
}
__device__ __forceinline__ void two_prod(float a, float b, float& p, float& e) {
    p = __fmul_rn(a, b);
    e = fmaf(a, b, -p);
}

// float-float squared norm of a point
__global__ void k_ff_norms(const float* __restrict__ X, long long n, int d, float2* __restrict__ N) {
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    float h = 0.f, l = 0.f;
    for (int c = 0; c < d; ++c) {
        const float x = X[i * d + c];
        float p, pe, s, e;
        two_prod(x, x, p, pe);
        two_sum(h, p, s, e);
        h = s;
        l = __fadd_rn(l, __fadd_rn(e, pe));
    }
    float s, e;
    fast_two_sum(h, l, s, e);
    N[i] = make_float2(s, e);
}

// A (FP64, nr columns) -> float-float pairs
__global__ void k_split64(const double* __restrict__ A, long long tot, float2* __restrict__ out) {
    const long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= tot) return;
    const double a = A[e];
    const float h = (float)a;
    out[e] = make_float2(h, (float)(a - (double)h));
}

constexpr int FF_THREADS = 128;
constexpr int FF_BN = 64;
constexpr float LN2_H = 0.693147182464599609375f;          // float nearest ln 2
constexpr float LN2_L = -1.904654323148236e-09f;           // ln 2 - LN2_H

// 2^(j/64), j = -32..32, as float-float pairs; a kernel argument (no copy or wait per call)
struct FfTab {
    float2 v[65];
};
static const FfTab& ff_table() {
    static const FfTab t = [] {
        FfTab h;
        for (int j = -32; j <= 32; ++j) {
            const double v = std::exp2(j / 64.0);
            const float hi = (float)v;
            h.v[j + 32] = make_float2(hi, (float)(v - (double)hi));
        }
        return h;
    }();
    return t;
}

// w_ij = K_ij (MODE 0) or t K_ij (MODE 1) as a float-float; false when K_ij < 2^-120, which is below
// any residual that matters.
template <int D, int MODE>
__device__ __forceinline__ bool ff_value(const float* xi, float2 ni, const float* xj, float2 nj, float sh, float sl,
                                         const float2* stab, float& Kh, float& Kl) {
    // x_i . x_j exactly up to the float-float accumulation
    float H = 0.f, L = 0.f;
#pragma unroll
    for (int c = 0; c < D; ++c) {
        float p, pe, s, e;
        two_prod(xi[c], xj[c], p, pe);
        two_sum(H, p, s, e);
        H = s;
        L = __fadd_rn(L, __fadd_rn(e, pe));
    }
    // D2 = n_i + n_j - 2 dot
    float A, a, B, b, Dh, Dl;
    two_sum(ni.x, nj.x, A, a);
    a = __fadd_rn(a, __fadd_rn(ni.y, nj.y));
    two_sum(A, -2.f * H, B, b);
    b = __fadd_rn(b, __fsub_rn(a, 2.f * L));
    fast_two_sum(B, b, Dh, Dl);
    if (Dh <= 0.f) Dh = 0.f, Dl = 0.f;
    // t = -s D2
    float th = __fmul_rn(-sh, Dh);
    float tl = fmaf(-sh, Dh, -th);
    tl = __fsub_rn(tl, __fadd_rn(__fmul_rn(sh, Dl), __fmul_rn(sl, Dh)));
    fast_two_sum(th, tl, th, tl);
    if (th < -120.f) return false;
    // 2^t = 2^m 2^(jj/64) e^z
    const float m = rintf(th);
    const float f64 = __fmul_rn(__fsub_rn(th, m), 64.f);
    const float jj = rintf(f64);
    const float r = __fmul_rn(__fsub_rn(f64, jj), 0.015625f);
    const float zh = __fmul_rn(r, LN2_H);
    const float zl = __fadd_rn(fmaf(r, LN2_H, -zh), __fadd_rn(__fmul_rn(r, LN2_L), __fmul_rn(tl, LN2_H)));
    const float q = __fmul_rn(__fmul_rn(zh, zh),
                              fmaf(zh, fmaf(zh, fmaf(zh, 1.f / 120.f, 1.f / 24.f), 1.f / 6.f), 0.5f));
    float Eh, El;
    fast_two_sum(1.f, zh, Eh, El);
    El = __fadd_rn(El, q);
    El = fmaf(Eh, zl, El);
    const float2 T = stab[(int)jj + 32];
    Kh = __fmul_rn(T.x, Eh);
    Kl = __fadd_rn(fmaf(T.x, Eh, -Kh), __fadd_rn(__fmul_rn(T.x, El), __fmul_rn(T.y, Eh)));
    fast_two_sum(Kh, Kl, Kh, Kl);
    const float sc = __int_as_float(((int)m + 127) << 23);   // 2^m, m in [-120, 0]
    Kh = __fmul_rn(Kh, sc);
    Kl = __fmul_rn(Kl, sc);
    if (MODE == 1) {   // w = t K
        const float ph = __fmul_rn(th, Kh);
        const float pl = __fadd_rn(fmaf(th, Kh, -ph), __fadd_rn(__fmul_rn(th, Kl), __fmul_rn(tl, Kh)));
        fast_two_sum(ph, pl, Kh, Kl);
    }
    return true;
}

// (Sh, Sl) += (Kh + Kl) (a.x + a.y)
__device__ __forceinline__ void ff_muladd(float Kh, float Kl, float2 a, float& Sh, float& Sl) {
    float p, pe, s, e;
    two_prod(Kh, a.x, p, pe);
    pe = __fadd_rn(pe, __fadd_rn(__fmul_rn(Kh, a.y), __fmul_rn(Kl, a.x)));
    two_sum(Sh, p, s, e);
    Sh = s;
    Sl = __fadd_rn(Sl, __fadd_rn(e, pe));
}

// Row block against column tiles: S_i = sum_j w_ij A_j in float-float, with w = K (mode 0)
// or w = t K, t = -s ||x_i - x_j||^2 in log2 units (mode 1, the sigma derivative up to -2 ln 2).
template <int D, int NR, int MODE>
__global__ void __launch_bounds__(FF_THREADS, 4)
k_rect_ff(const float* __restrict__ Xr, int nr, const float2* __restrict__ NR_, const float* __restrict__ Xc,
          int nc, const float2* __restrict__ NC_, float sh, float sl, const float2* __restrict__ Aff,
          const FfTab tab, int tiles_per_split, double* __restrict__ part) {
    __shared__ float sx[FF_BN][D + 1];
    __shared__ float2 snrm[FF_BN];
    __shared__ float2 sa[NR][FF_BN];
    __shared__ float2 stab[65];
    const int tid = threadIdx.x;
    if (tid < 65) stab[tid] = tab.v[tid];
    const long long i = (long long)blockIdx.x * FF_THREADS + tid;
    const bool row_ok = i < nr;
    float xi[D];
#pragma unroll
    for (int c = 0; c < D; ++c) xi[c] = row_ok ? Xr[i * D + c] : 0.f;
    const float2 ni = row_ok ? NR_[i] : make_float2(0.f, 0.f);
    double acc[NR];
#pragma unroll
    for (int q = 0; q < NR; ++q) acc[q] = 0.0;

    const int ntiles = (nc + FF_BN - 1) / FF_BN;
    const int t0 = blockIdx.y * tiles_per_split;
    const int t1 = min(t0 + tiles_per_split, ntiles);
    for (int t = t0; t < t1; ++t) {
        const int c0 = t * FF_BN;
        __syncthreads();
        for (int e = tid; e < FF_BN * D; e += FF_THREADS) {
            const int j = e / D, c = e - j * D;
            sx[j][c] = (c0 + j < nc) ? Xc[(size_t)(c0 + j) * D + c] : 0.f;
        }
        for (int e = tid; e < FF_BN; e += FF_THREADS)
            snrm[e] = (c0 + e < nc) ? NC_[c0 + e] : make_float2(0.f, 0.f);
        for (int e = tid; e < NR * FF_BN; e += FF_THREADS) {
            const int q = e / FF_BN, j = e - q * FF_BN;
            sa[q][j] = (c0 + j < nc) ? Aff[(size_t)q * nc + c0 + j] : make_float2(0.f, 0.f);
        }
        __syncthreads();
        float Sh[NR], Sl[NR];
#pragma unroll
        for (int q = 0; q < NR; ++q) Sh[q] = 0.f, Sl[q] = 0.f;
        const int jmax = min(FF_BN, nc - c0);
        for (int j = 0; j < jmax; ++j) {
            float Kh, Kl;
            if (!ff_value<D, MODE>(xi, ni, sx[j], snrm[j], sh, sl, stab, Kh, Kl)) continue;
#pragma unroll
            for (int qq = 0; qq < NR; ++qq) ff_muladd(Kh, Kl, sa[qq][j], Sh[qq], Sl[qq]);
        }
#pragma unroll
        for (int qq = 0; qq < NR; ++qq) acc[qq] += (double)Sh[qq] + (double)Sl[qq];
    }
    if (row_ok) {
#pragma unroll
        for (int q = 0; q < NR; ++q) part[((size_t)blockIdx.y * NR + q) * nr + i] = acc[q];
    }
}

// ------------------------------------------------------------------ one point set, one column
// The same sums over one point set: w_ij is symmetric, so a pair i < j is evaluated once and serves
// both S_i and S_j (about 150 FP32 operations for w at d = 8 against 14 for each sum).  The order of
// work and its split are those of sym_tc.cu.  The lanes of a warp are 8 row groups x 4 column
// groups; a thread holds R rows and takes one column at a time.  Sums are float-float over one
// column tile (rows) or over R rows, 8 lanes (columns), and FP64 beyond, as above.
// R = 4, 2 or 1: units of 256 x 128, 128 x 128 or 64 x 64 pairs, so that small sets fill the chip.
// Measured (one residual, against k_rect_ff): n = 30011, d = 8 2.90 ms against 5.00 (71% of the FMA
// pipe's rate, 2.06 ms for the operations above), n = 10^5 30.9 against 55 ms.
template <int R>
constexpr int sff_bn() { return R == 1 ? 64 : 128; }
constexpr int SFF_T = 256, SFF_NW = SFF_T / 32;

template <int D, int MODE, int R, class Grid>
__global__ void __launch_bounds__(SFF_T, 2)
k_sym_ff(const float* __restrict__ X, Grid sg, const float2* __restrict__ N2, float sh, float sl,
         const float2* __restrict__ Aff, const FfTab tab, double* __restrict__ rowpart,
         double* __restrict__ colpart) {
    constexpr int BN = sff_bn<R>(), RB = 8 * SFF_NW * R;
    __shared__ float sx[BN][D + (D % 2 == 0)];     // odd stride: the four columns in different banks
    __shared__ float2 snrm[BN], sa[BN], stab[65];
    __shared__ float2 sC[2][SFF_NW][BN];
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    const int lr = lane & 7, lc = lane >> 3;
    if (tid < 65) stab[tid] = tab.v[tid];
    const int run = blockIdx.x;
    int u = (int)sg.run_begin(run);
    const int u1 = (int)sg.run_begin(run + 1);
    int I = sg.block_of(u), cc = 0;
    long long at = -1;                             // where the last unit's column sums go
    auto store_column = [&](int b) {
        if (at >= 0 && tid < BN) {
            double x = 0.0;
#pragma unroll
            for (int k = 0; k < SFF_NW; ++k) {
                const float2 c = sC[b][k][tid];
                x += (double)c.x + (double)c.y;
            }
            colpart[at + tid] = x;
        }
    };
    for (; u < u1; ++I) {
        const int uI = (int)sg.first(I), ue = min(u1, (int)sg.first(I + 1));
        float xi[R][D];
        float2 ni[R], ai[R];
        double acc[R];
#pragma unroll
        for (int r = 0; r < R; ++r) {
            const long long row = (long long)I * RB + w * 8 * R + 8 * r + lr;
            const bool ok = row < sg.n;
#pragma unroll
            for (int c = 0; c < D; ++c) xi[r][c] = ok ? X[row * D + c] : 0.f;
            ni[r] = ok ? N2[row] : make_float2(0.f, 0.f);
            ai[r] = ok ? Aff[row] : make_float2(0.f, 0.f);
            acc[r] = 0.0;
        }
        for (; u < ue; ++u, ++cc) {
            const int T = I * sg.RU + (u - uI), b = cc & 1;
            const long long c0 = (long long)T * BN;
            __syncthreads();                       // the tile before is consumed
            store_column(b ^ 1);
            for (int e = tid; e < BN * D; e += SFF_T) {
                const int j = e / D, c = e - j * D;
                sx[j][c] = c0 + j < sg.n ? X[c0 * D + e] : 0.f;
            }
            for (int e = tid; e < BN; e += SFF_T) {
                const bool ok = c0 + e < sg.n;
                snrm[e] = ok ? N2[c0 + e] : make_float2(0.f, 0.f);
                sa[e] = ok ? Aff[c0 + e] : make_float2(0.f, 0.f);   // padding adds nothing
            }
            __syncthreads();
            float Sh[R], Sl[R];
#pragma unroll
            for (int r = 0; r < R; ++r) Sh[r] = Sl[r] = 0.f;
#pragma unroll 1
            for (int k = 0; k < BN / 4; ++k) {
                const int j = 4 * k + lc;
                float xj[D];
#pragma unroll
                for (int c = 0; c < D; ++c) xj[c] = sx[j][c];
                const float2 nj = snrm[j], aj = sa[j];
                float ch = 0.f, cl = 0.f;
#pragma unroll
                for (int r = 0; r < R; ++r) {
                    float Kh, Kl;
                    if (ff_value<D, MODE>(xi[r], ni[r], xj, nj, sh, sl, stab, Kh, Kl)) {
                        ff_muladd(Kh, Kl, aj, Sh[r], Sl[r]);
                        ff_muladd(Kh, Kl, ai[r], ch, cl);
                    }
                }
                __syncwarp();
#pragma unroll
                for (int st = 1; st <= 4; st <<= 1) {
                    const float oh = __shfl_xor_sync(0xffffffffu, ch, st), ol = __shfl_xor_sync(0xffffffffu, cl, st);
                    float s, e;
                    two_sum(ch, oh, s, e);
                    ch = s;
                    cl = __fadd_rn(__fadd_rn(cl, ol), e);
                }
                if (lr == 0) sC[b][w][j] = make_float2(ch, cl);
            }
#pragma unroll
            for (int r = 0; r < R; ++r) acc[r] += (double)Sh[r] + (double)Sl[r];
            at = T / sg.RU > I ? sg.col_base(T) + (long long)sg.slot(I) * BN : -1;
        }
#pragma unroll
        for (int r = 0; r < R; ++r) {              // over the four column groups
            double x = acc[r];
            x += __shfl_xor_sync(0xffffffffu, x, 8);
            x += __shfl_xor_sync(0xffffffffu, x, 16);
            if (lc == 0) rowpart[(long long)(run + sg.slot(I)) * RB + w * 8 * R + 8 * r + lr] = x;
        }
    }
    __syncthreads();
    store_column((cc & 1) ^ 1);
}

// Point i's slots in a fixed order; out = scale S (Y null) or Y - beta A - S.  With panels acc holds the
// sums of those before, and out is written after the last.
template <class Grid>
__global__ void __launch_bounds__(256)
k_sym_ff_reduce(Grid sg, const double* __restrict__ rowpart, const double* __restrict__ colpart, double scale,
                const float* __restrict__ Y, const double* __restrict__ A, double beta, double* __restrict__ out,
                double* __restrict__ acc) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= sg.n) return;
    const int T = i / sg.BN, b = T / sg.RU;
    const double* cp = colpart + sg.col_base(T) + i % sg.BN;
    double s = 0.0;
#pragma unroll 4
    for (int I = 0; I < sg.slots(b); ++I) s += cp[(long long)I * sg.BN];
    if (sg.has(b)) {
        const int s0 = sg.run_of(sg.first(b)), s1 = sg.run_of(sg.first(b + 1) - 1);
        for (int r = s0; r <= s1; ++r) s += rowpart[(long long)(r + sg.slot(b)) * sg.rows() + i % sg.rows()];
    }
    if (!sg.first_panel()) s += acc[i];
    if (!sg.last_panel()) {
        acc[i] = s;
        return;
    }
    out[i] = Y ? (double)Y[i] - beta * A[i] - s : scale * s;
}

template <class Grid>
using sff_fn = void (*)(const float*, Grid, const float2*, float, float, const float2*, FfTab, double*, double*);
template <int D, class Grid>
static sff_fn<Grid> sff_pick1(int mode, int R) {
    if (R == 4) return mode == 0 ? &k_sym_ff<D, 0, 4, Grid> : &k_sym_ff<D, 1, 4, Grid>;
    if constexpr (std::is_same<Grid, SyGrid>::value) {   // panels are for large sets, with four rows
        if (mode == 0) return R == 2 ? &k_sym_ff<D, 0, 2, Grid> : &k_sym_ff<D, 0, 1, Grid>;
        return R == 2 ? &k_sym_ff<D, 1, 2, Grid> : &k_sym_ff<D, 1, 1, Grid>;
    }
    return nullptr;
}
template <class Grid>
static sff_fn<Grid> sff_pick(int d, int mode, int R) {
    switch (d) {
#define KRR_D(v) \
    case v: return sff_pick1<v, Grid>(mode, R);
        KRR_D(1) KRR_D(2) KRR_D(3) KRR_D(4) KRR_D(5) KRR_D(6) KRR_D(7) KRR_D(8)
        KRR_D(9) KRR_D(10) KRR_D(11) KRR_D(12) KRR_D(13) KRR_D(14) KRR_D(15) KRR_D(16)
#undef KRR_D
    }
    return nullptr;
}

__global__ void k_rect_ff_reduce(const double* __restrict__ part, int splits, int n, int nr,
                                 double scale, double* __restrict__ out) {
    const long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= (long long)n * nr) return;
    const int q = (int)(e / n);
    const int i = (int)(e - (long long)q * n);
    double s = 0.0;
    for (int sp = 0; sp < splits; ++sp) s += part[((size_t)sp * nr + q) * n + i];
    out[(size_t)q * n + i] = scale * s;
}

__global__ void k_resid_ff_reduce(const double* __restrict__ part, int splits, int n, int nr,
                                  const float* __restrict__ Y, const double* __restrict__ A,
                                  double beta, double* __restrict__ R) {
    const long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= (long long)n * nr) return;
    const int q = (int)(e / n);
    const int i = (int)(e - (long long)q * n);
    double s = 0.0;
    for (int sp = 0; sp < splits; ++sp) s += part[((size_t)sp * nr + q) * n + i];
    R[(size_t)q * n + i] = (double)Y[(size_t)q * n + i] - beta * A[(size_t)q * n + i] - s;
}

typedef void (*ff_fn)(const float*, int, const float2*, const float*, int, const float2*, float, float,
                      const float2*, FfTab, int, double*);

template <int D, int MODE>
static ff_fn ff_pick1(int nr) {
    switch (nr) {
        case 1: return &k_rect_ff<D, 1, MODE>;
        case 2: return MODE == 0 ? &k_rect_ff<D, 2, MODE> : nullptr;
        case 4: return MODE == 0 ? &k_rect_ff<D, 4, MODE> : nullptr;
        case 8: return MODE == 0 ? &k_rect_ff<D, 8, MODE> : nullptr;
        case 16: return MODE == 0 ? &k_rect_ff<D, 16, MODE> : nullptr;
    }
    return nullptr;
}

static ff_fn ff_pick(int d, int nr, int mode) {
    switch (d) {
#define KRR_D(v) \
    case v: return mode == 0 ? ff_pick1<v, 0>(nr) : ff_pick1<v, 1>(nr);
        KRR_D(1) KRR_D(2) KRR_D(3) KRR_D(4) KRR_D(5) KRR_D(6) KRR_D(7) KRR_D(8)
        KRR_D(9) KRR_D(10) KRR_D(11) KRR_D(12) KRR_D(13) KRR_D(14) KRR_D(15) KRR_D(16)
#undef KRR_D
    }
    return nullptr;
}

int choose_splits_public(int nblk, int ntiles, int slots);

// part (splits x nrhs x nr) of S_i = sum_j w_ij A_j for rows Xr and columns Xc (mode as above).
static int rect_ff_parts(krr_ctx* ctx, const float* Xr, long long nr, const float* Xc, long long nc,
                         int d, double sigma, const double* A, int nrhs_chunk, int mode,
                         double** part_out, int* splits_out) {
    const FfTab& tab = ff_table();
    float2 *NXr, *NXc, *Aff;
    KRR_RET(bufT(ctx, "ff_nr", (size_t)nr, &NXr));
    KRR_RET(bufT(ctx, "ff_nc", (size_t)nc, &NXc));
    KRR_RET(bufT(ctx, "ff_alpha", (size_t)nc * nrhs_chunk, &Aff));
    k_ff_norms<<<ceil_div(nr, 256), 256, 0, ctx->stream>>>(Xr, nr, d, NXr);
    KRR_CHECK_LAUNCH();
    k_ff_norms<<<ceil_div(nc, 256), 256, 0, ctx->stream>>>(Xc, nc, d, NXc);
    KRR_CHECK_LAUNCH();
    k_split64<<<ceil_div(nc * nrhs_chunk, 256), 256, 0, ctx->stream>>>(A, nc * nrhs_chunk, Aff);
    KRR_CHECK_LAUNCH();
    const double s = 1.4426950408889634 / (2.0 * sigma * sigma);
    const float sh = (float)s, sl = (float)(s - (double)sh);
    ff_fn fn = ff_pick(d, nrhs_chunk, mode);
    if (!fn) return fail(ctx, KRR_E_INVAL, "float-float product: unsupported shape");
    const int nblk = (int)ceil_div(nr, FF_THREADS);
    const int ntiles = (int)ceil_div(nc, FF_BN);
    int occ = 1;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, (const void*)fn, FF_THREADS, 0);
    const int slots = ctx->num_sms * std::max(occ, 1);
    int splits = choose_splits_public(nblk, ntiles, slots);
    const int tps = (ntiles + splits - 1) / splits;
    splits = (ntiles + tps - 1) / tps;
    double* part;
    KRR_RET(bufT(ctx, "ff_part", (size_t)splits * nrhs_chunk * nr, &part));
    dim3 grid(nblk, splits);
    fn<<<grid, FF_THREADS, 0, ctx->stream>>>(Xr, (int)nr, NXr, Xc, (int)nc, NXc, sh, sl, Aff, tab, tps, part);
    KRR_CHECK_LAUNCH();
    *part_out = part;
    *splits_out = splits;
    return KRR_OK;
}

int kernel_occupancy(const void* fn, int threads);   // kmvm.cu

// One column over one point set (see k_sym_ff).  *ran is false, with nothing launched, where the
// partial sums do not fit the device or the set is too large for the form.
static int sym_ff(krr_ctx* ctx, const float* X, long long n, int d, double sigma, const double* A, int mode,
                  double out_scale, const float* Y, double beta, double* out, bool* ran) {
    *ran = false;
    if (n > (1LL << 19)) return KRR_OK;
    SyGrid g{}, best{};
    int bestR = 0;
    double best_cost = 0.0;
    for (int R = 4; R >= 1; R /= 2) {
        const sff_fn<SyGrid> f = sff_pick<SyGrid>(d, mode, R);
        if (!f) return fail(ctx, KRR_E_INVAL, "float-float product: unsupported shape");
        const int RB = 8 * SFF_NW * R;
        g.n = (int)n;
        g.BN = R == 1 ? 64 : 128;
        g.RU = RB / g.BN;
        g.NU = (int)ceil_div(n, RB) * g.RU;
        g.nblk = g.NU / g.RU;
        g.W = g.first(g.nblk);
        g.G = (int)std::min<long long>(g.W, (long long)ctx->num_sms * kernel_occupancy((const void*)f, SFF_T));
        // the longest run sets the time: units x (pairs, and a column's lane sum per R rows)
        const double cost = (double)((g.W + g.G - 1) / g.G) * RB * g.BN * (1.0 + 0.2 / R) *
                            ((g.G + ctx->num_sms - 1) / ctx->num_sms);
        if (8 * g.col_base(g.NU) > kSymBytes && R < 4) break;   // panels have four rows
        if (!bestR || cost < best_cost) {
            best_cost = cost;
            best = g;
            bestR = R;
        }
    }
    g = best;
    float2 *N2, *Aff;
    double* acc = nullptr;
    if (8 * g.col_base(g.NU) > kSymBytes) KRR_RET(bufT(ctx, "sym_acc", (size_t)n, &acc));
    KRR_RET(bufT(ctx, "ff_nr", (size_t)n, &N2));
    KRR_RET(bufT(ctx, "ff_alpha", (size_t)n, &Aff));
    const double s = 1.4426950408889634 / (2.0 * sigma * sigma);
    const float sh = (float)s, sl = (float)(s - (double)sh);
    bool split = false;
    const int rc = sym_product(ctx, g, [&](const auto& p, void* row, void* col) -> int {
        using Grid = std::decay_t<decltype(p)>;
        double *rowpart = (double*)row, *colpart = (double*)col;
        if (!split) {
            k_ff_norms<<<ceil_div(n, 256), 256, 0, ctx->stream>>>(X, n, d, N2);
            KRR_CHECK_LAUNCH();
            k_split64<<<ceil_div(n, 256), 256, 0, ctx->stream>>>(A, n, Aff);
            KRR_CHECK_LAUNCH();
            split = true;
        }
        sff_pick<Grid>(d, mode, bestR)<<<p.G, SFF_T, 0, ctx->stream>>>(X, p, N2, sh, sl, Aff, ff_table(), rowpart, colpart);
        KRR_CHECK_LAUNCH();
        k_sym_ff_reduce<Grid><<<ceil_div(n, 256), 256, 0, ctx->stream>>>(p, rowpart, colpart, out_scale, Y, A, beta, out,
                                                                         acc);
        KRR_CHECK_LAUNCH();
        return KRR_OK;
    });
    if (rc == KRR_E_NOMEM) {                       // of sym_buffers, before any launch
        ctx->err.clear();
        return KRR_OK;
    }
    KRR_RET(rc);
    *ran = true;
    return KRR_OK;
}

int launch_residual_ff(krr_ctx* ctx, const float* X, long long n, int d, double sigma, double beta,
                       const float* Y, const double* A, int nrhs, double* R) {
    if (n > 0x7fffffffLL) return fail(ctx, KRR_E_INVAL, "residual: more than 2^31 points");
    if (d > 16) return launch_residual_hp(ctx, X, n, d, sigma, beta, Y, A, nrhs, R);
    int done = 0;
    while (done < nrhs) {
        const int left = nrhs - done;
        const int chunk = left >= 16 ? 16 : left >= 8 ? 8 : left >= 4 ? 4 : left >= 2 ? 2 : 1;
        if (chunk == 1) {
            bool ran;
            KRR_RET(sym_ff(ctx, X, n, d, sigma, A + (size_t)done * n, 0, 1.0, Y + (size_t)done * n, beta,
                           R + (size_t)done * n, &ran));
            if (ran) {
                done += chunk;
                continue;
            }
        }
        double* part;
        int splits;
        KRR_RET(rect_ff_parts(ctx, X, n, X, n, d, sigma, A + (size_t)done * n, chunk, 0, &part, &splits));
        k_resid_ff_reduce<<<ceil_div(n * chunk, 256), 256, 0, ctx->stream>>>(
            part, splits, (int)n, chunk, Y + (size_t)done * n, A + (size_t)done * n, beta,
            R + (size_t)done * n);
        KRR_CHECK_LAUNCH();
        done += chunk;
    }
    return KRR_OK;
}

// out (nr) = K(Xr, Xc) a (mode 0) or (dK(Xr, Xc)/dlog sigma) a (mode 1), float-float, FP64 in/out.
int launch_rect_ff(krr_ctx* ctx, const float* Xr, long long nr, const float* Xc, long long nc, int d,
                   double sigma, const double* a, int mode, double* out) {
    if (nr > 0x7fffffffLL || nc > 0x7fffffffLL) return fail(ctx, KRR_E_INVAL, "too many points");
    if (d > 16) return fail(ctx, KRR_E_INVAL, "float-float products need d <= 16");
    const double scale = mode == 1 ? -2.0 * 0.6931471805599453 : 1.0;
    if (Xr == Xc && nr == nc) {
        bool ran;
        KRR_RET(sym_ff(ctx, Xr, nr, d, sigma, a, mode, scale, nullptr, 0.0, out, &ran));
        if (ran) return KRR_OK;
    }
    double* part;
    int splits;
    KRR_RET(rect_ff_parts(ctx, Xr, nr, Xc, nc, d, sigma, a, 1, mode, &part, &splits));
    k_rect_ff_reduce<<<ceil_div(nr, 256), 256, 0, ctx->stream>>>(part, splits, (int)nr, 1, scale, out);
    KRR_CHECK_LAUNCH();
    return KRR_OK;
}

}  // namespace krr

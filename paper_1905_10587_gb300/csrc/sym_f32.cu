// Symmetric FP32 product: Q = (K(X, X) + beta I) v for one right-hand side on the expansion or on
// exact coordinate differences, with every kernel value of a pair i < j evaluated once.
//
// k_kmvm2 is bound by the FMA pipe: D + 1 (expansion) or 2 D + 1 (differences) operations for the
// exponent of each of the n^2 entries, and one more for the sum.  Here an entry right of the
// diagonal blocks adds to both q_i and q_j, which halves the exponents for one more FMA.
//
// A thread holds R rows; the lanes of a warp are 8 row groups x 4 column groups (a quarter warp
// shares a column, so that its 16-byte shared load is one address), so that a warp has 8 R rows and
// takes four columns at a time, each thread one.  Per column a thread adds its R
// entries to R row sums (registers, folded float-float every tile) and to one column sum; eight
// column sums are then reduced over the eight row groups with 7 shuffles, the same ~4
// instructions per column that any number of row groups would need, but with 8 registers instead
// of 32.  Rows go two at a time through the paired FP32 instructions, columns are staged in
// shared memory with every value duplicated (one shared load feeds both halves), two tiles deep
// with the next tile's global loads in flight.
//
// R = 8 with four warps or R = 4 with eight; a row block is 256 rows in both.  Work order, split and
// partial sums are those of sym_tc.cu.
//
// Measured against k_kmvm2 (us per krr_kmvm call): expansion n = 30011 d = 6 221 against 367,
// n = 10^5 d = 8 2475 against 3823; differences n = 30011 d = 12 533 against 787; at n <= 2000 both are
// the call's ~25 us of launches.  It runs at 56-65% of the FMA pipe; shared loads and lane sums take
// most of the other issue slots.
#include "internal.cuh"
#include "sym.cuh"

#include <algorithm>
#include <type_traits>

namespace krr {

constexpr int SF_ROWS = 256;                       // rows per block

__device__ __forceinline__ unsigned long long sf_fma(unsigned long long a, unsigned long long b,
                                                     unsigned long long c) {
    unsigned long long d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}
__device__ __forceinline__ unsigned long long sf_add(unsigned long long a, unsigned long long b) {
    unsigned long long d;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ unsigned long long sf_sub(unsigned long long a, unsigned long long b) {
    unsigned long long d;
    asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ unsigned long long sf_mul(unsigned long long a, unsigned long long b) {
    unsigned long long d;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}

// RAW as for k_kmvm2: P holds the caller's coordinates and the exponent is nsc ||x_i - x_j||^2.
template <int D, int R, bool RAW, class Grid>
__global__ void __launch_bounds__(SF_ROWS / R * 4)
k_sym_f32(const float* __restrict__ P, Grid sg, const float* __restrict__ V, float nsc,
          float2* __restrict__ rowpart, float2* __restrict__ colpart) {
    pdl_entry();
    constexpr int NT = SF_ROWS / R * 4;            // threads
    constexpr int NW = NT / 32;
    constexpr int PS = (D + 1 + 3) / 4 * 4;
    constexpr int NV = D + (RAW ? 1 : 2);          // staged values per column: coordinates, norm, v
    constexpr int SW = (NV + 1) / 2 | 1;           // 16-byte words per column; odd: four neighbouring
                                                   // columns sit in different banks
    constexpr int RP = R / 2;
    constexpr int TL = SY_T * PS / 4 / NT + (SY_T * PS / 4 % NT != 0);   // float4s of a tile per thread
    __shared__ __align__(16) ulonglong2 sP[2][SY_T * SW];
    __shared__ float sC[2][NW][SY_T];
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    const int lr = lane & 7, lc = lane >> 3;
    const float4* P4 = reinterpret_cast<const float4*>(P);
    const int run = blockIdx.x;
    int u = (int)sg.run_begin(run);
    const int u1 = (int)sg.run_begin(run + 1);
    int I = sg.block_of(u);
    const unsigned long long nsc2 = sy_pack(nsc, nsc);

    // the tile in flight: packed points and v of SY_T columns
    float4 g[TL];
    float gv = 0.f;
    auto fetch = [&](int T) {
#pragma unroll
        for (int e = 0; e < TL; ++e) {
            const int f = tid + e * NT, j = f / (PS / 4);
            g[e] = make_float4(0.f, 0.f, 0.f, 0.f);
            if (f < SY_T * PS / 4 && T * SY_T + j < sg.n) g[e] = P4[(size_t)T * SY_T * (PS / 4) + f];
        }
        if (tid < SY_T) gv = T * SY_T + tid < sg.n ? V[T * SY_T + tid] : 0.f;
    };
    auto stage = [&](int b) {
        unsigned long long* s = reinterpret_cast<unsigned long long*>(sP[b]);
#pragma unroll
        for (int e = 0; e < TL; ++e) {
            const int f = tid + e * NT, j = f / (PS / 4), c0 = 4 * (f - j * (PS / 4));
            if (f >= SY_T * PS / 4) break;
            const float x[4] = {g[e].x, g[e].y, g[e].z, g[e].w};
#pragma unroll
            for (int k = 0; k < 4; ++k)
                if (c0 + k < NV - 1) s[j * (2 * SW) + c0 + k] = sy_pack(x[k], x[k]);
        }
        if (tid < SY_T) s[tid * (2 * SW) + NV - 1] = sy_pack(gv, gv);
    };
    // column sums of the unit before, over the warps
    long long at = -1;
    auto store_column = [&](int b) {
        if (at >= 0 && tid < SY_T) {
            float2 x = make_float2(0.f, 0.f);
#pragma unroll
            for (int k = 0; k < NW; ++k) ff_add(x.x, x.y, sC[b][k][tid]);
            colpart[at + tid] = x;
        }
    };

    const int T0 = I * sg.RU + (u - (int)sg.first(I));
    fetch(T0);
    stage(0);
    int cc = 0;
    while (u < u1) {
        const int uI = (int)sg.first(I), ue = min(u1, (int)sg.first(I + 1));
        // this thread's rows: lr + 8 k of the warp's 8 R
        unsigned long long xi[RP][D], ai[RP], vi[RP], acc[RP];
        float fh[R], fl[R];
#pragma unroll
        for (int p = 0; p < RP; ++p) {
            float x[2][PS], v[2];
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int row = I * SF_ROWS + w * 8 * R + lr + 8 * (2 * p + h);
                const bool ok = row < sg.n;
                v[h] = ok ? V[row] : 0.f;
#pragma unroll
                for (int c = 0; c < PS / 4; ++c) {
                    const float4 t = ok ? P4[(size_t)row * (PS / 4) + c] : make_float4(0.f, 0.f, 0.f, 0.f);
                    x[h][4 * c] = t.x;
                    x[h][4 * c + 1] = t.y;
                    x[h][4 * c + 2] = t.z;
                    x[h][4 * c + 3] = t.w;
                }
            }
#pragma unroll
            for (int c = 0; c < D; ++c)
                xi[p][c] = RAW ? sy_pack(x[0][c], x[1][c]) : sy_pack(2.f * x[0][c], 2.f * x[1][c]);
            ai[p] = sy_pack(x[0][D], x[1][D]);
            vi[p] = sy_pack(v[0], v[1]);
        }
#pragma unroll
        for (int r = 0; r < R; ++r) fh[r] = fl[r] = 0.f;
        for (; u < ue; ++u, ++cc) {
            const int T = I * sg.RU + (u - uI), b = cc & 1;
            // One barrier a tile: behind it this tile is staged, the other tile buffer and the
            // column sums of the tile before are free to use.
            __syncthreads();
            store_column(b ^ 1);
            const bool more = u + 1 < u1;
            // the next pair is the next column tile, or the next block's first
            if (more) fetch(u + 1 < ue ? T + 1 : (I + 1) * sg.RU);
#pragma unroll
            for (int p = 0; p < RP; ++p) acc[p] = 0ull;
#pragma unroll 1
            for (int q = 0; q < SY_T / 32; ++q) {
                float cs[8];
#pragma unroll
                for (int k = 0; k < 8; ++k) {
                    const ulonglong2* s = sP[b] + (32 * q + 4 * k + lc) * SW;
                    unsigned long long xj[2 * SW];
#pragma unroll
                    for (int e = 0; e < (NV + 1) / 2; ++e) {
                        const ulonglong2 t = s[e];
                        xj[2 * e] = t.x;
                        xj[2 * e + 1] = t.y;
                    }
                    unsigned long long c2 = 0ull;
#pragma unroll
                    for (int p = 0; p < RP; ++p) {
                        unsigned long long tt;
                        if constexpr (RAW) {
                            unsigned long long ss = 0ull;
#pragma unroll
                            for (int c = 0; c < D; ++c) {
                                const unsigned long long df = sf_sub(xi[p][c], xj[c]);
                                ss = sf_fma(df, df, ss);
                            }
                            tt = sf_mul(ss, nsc2);
                        } else {
                            tt = sf_add(ai[p], xj[D]);
#pragma unroll
                            for (int c = 0; c < D; ++c) tt = sf_fma(xi[p][c], xj[c], tt);
                        }
                        float t0, t1;
                        sy_unpack(tt, t0, t1);
                        const unsigned long long e = sy_pack(ex2f(t0), ex2f(t1));
                        sy_fma(acc[p], e, xj[NV - 1]);
                        sy_fma(c2, e, vi[p]);
                    }
                    float lo, hi;
                    sy_unpack(c2, lo, hi);
                    cs[k] = lo + hi;
                }
                // over the row groups: lane (lr, lc) ends with column 4 lr + lc of the 32
                lane_sum<8, 4>(cs, lane);
                sC[b][w][32 * q + 4 * lr + lc] = cs[0];
            }
#pragma unroll
            for (int p = 0; p < RP; ++p) {
                float lo, hi;
                sy_unpack(acc[p], lo, hi);
                ff_add(fh[2 * p], fl[2 * p], lo);
                ff_add(fh[2 * p + 1], fl[2 * p + 1], hi);
            }
            if (more) stage(b ^ 1);
            // inside the diagonal block both triangles were evaluated: row sums only
            at = T / sg.RU > I ? sg.col_base(T) + (long long)sg.slot(I) * SY_T : -1;
        }
        // the piece's row sums, over the four column groups
#pragma unroll
        for (int r = 0; r < R; ++r) {
            float h = fh[r], l = fl[r];
#pragma unroll
            for (int st = 8; st <= 16; st <<= 1) {
                const float oh = __shfl_xor_sync(0xffffffffu, h, st), ol = __shfl_xor_sync(0xffffffffu, l, st);
                ff_add(h, l, oh);
                l += ol;
            }
            if (lc == 0) rowpart[(long long)(run + sg.slot(I)) * SF_ROWS + w * 8 * R + lr + 8 * r] = make_float2(h, l);
        }
        ++I;
    }
    __syncthreads();
    store_column((cc & 1) ^ 1);
}

template <class Grid>
using sf_fn = void (*)(const float*, Grid, const float*, float, float2*, float2*);

// Eight rows per thread halve the shared loads and lane sums per entry, at up to 254 registers (two
// blocks a SM).  Measured at n = 30011 (us, whole call): expansion d = 12 326 against 352 with four
// rows, d = 16 405 against 472; differences, bound by their longer FMA chains, d = 12 527 against 533,
// d = 16 747 against 726, and at n = 8000 80 against 72, so they take four above d = 10.
template <int D, bool RAW>
constexpr int sf_rows() { return RAW && D > 10 ? 4 : 8; }
template <int D, class Grid>
static sf_fn<Grid> sf_pick1(bool raw, int* R) {
    *R = raw ? sf_rows<D, true>() : sf_rows<D, false>();
    return raw ? &k_sym_f32<D, sf_rows<D, true>(), true, Grid> : &k_sym_f32<D, sf_rows<D, false>(), false, Grid>;
}
template <class Grid>
static sf_fn<Grid> sf_pick(int dk, bool raw, int* R) {
    switch (dk) {
#define KRR_D(v) \
    case v: return sf_pick1<v, Grid>(raw, R);
        KRR_D(1) KRR_D(2) KRR_D(3) KRR_D(4) KRR_D(5) KRR_D(6) KRR_D(7) KRR_D(8)
        KRR_D(9) KRR_D(10) KRR_D(11) KRR_D(12) KRR_D(13) KRR_D(14) KRR_D(15) KRR_D(16)
#undef KRR_D
    }
    return nullptr;
}

int kernel_occupancy(const void* fn, int threads);   // kmvm.cu

// Whether the symmetric form takes a square product.
bool sym_f32_fits(long long n, int d) { return kernel_dim(d) <= 16 && n <= (1LL << 19); }

// Q = (K + beta I) V for packed points P (raw_nsc = 0) or raw coordinates (raw_nsc = -s).
int launch_kmvm_sym_f32(krr_ctx* ctx, const float* P, long long n, int d, float beta, const float* V, float* Q,
                        float raw_nsc) {
    int R = 8;
    const sf_fn<SyGrid> fn = sf_pick<SyGrid>(kernel_dim(d), raw_nsc != 0.f, &R);
    if (!fn) return fail(ctx, KRR_E_INVAL, "symmetric product: unsupported dimension");
    const int threads = SF_ROWS / R * 4;
    SyGrid g{};
    g.n = (int)n;
    g.BN = SY_T;
    g.RU = SF_ROWS / SY_T;
    g.NU = (int)ceil_div(n, SF_ROWS) * g.RU;
    g.nblk = g.NU / g.RU;
    g.W = g.first(g.nblk);
    g.G = (int)std::min<long long>(g.W, (long long)ctx->num_sms * kernel_occupancy((const void*)fn, threads));
    SyPoints pts;
    pts.P = P;
    pts.d = kernel_dim(d);
    pts.ps = packed_stride(d);
    pts.nsc = raw_nsc;
    return sym_product(ctx, g, [&](const auto& p, void* row, void* col) -> int {
        using Grid = std::decay_t<decltype(p)>;
        float2 *rowpart = (float2*)row, *colpart = (float2*)col;
        launch_pdl(sf_pick<Grid>(kernel_dim(d), raw_nsc != 0.f, &R), p.G, threads, 0, ctx->stream, P, p, V, raw_nsc, rowpart,
                   colpart);
        KRR_CHECK_LAUNCH();
        return launch_sym_reduce(ctx, p, rowpart, colpart, V, beta, 1.0, nullptr, Q, pts);
    });
}

}  // namespace krr

// Column-pivoted QR pivot selection (Algorithm 1, steps 3-4) on Y^T.
//
// The columns of Y^T are the rows of the n x l sketch Y.  Step m takes the row p whose
// residual (its part orthogonal to the rows chosen before) has the largest norm, lowest
// index on ties: the Businger-Golub pivot sequence.  The residuals are kept by
// Householder reflectors acting on the coordinates of the rows, blocked in panels of
// QH_B pivots:
//   * reflector m (coordinates m..l-1) is built from the pivot row's current residual,
//     H_m = I - tau_m v_m v_m^T with v_m[m] = 1;
//   * within a panel the rows are not rewritten: c[i][j] = tau_j v_j . y_i^(j) records
//     what reflector j does to row i, so y_i^(m) = y_i^(m0) - sum_j c[i][j] v_j, and one
//     read-only pass over the trailing coordinates m..l-1 per pivot gives c[i][m], the new
//     coordinate r_im of every row and its residual norm by downdating (FP64);
//   * at the end of a panel one pass applies the panel's reflectors to the coordinates
//     beyond it and recomputes every residual norm from them.
// Each pivot reads n x (l - m) floats (the trailing part shrinks), and each panel reads
// and writes it once, instead of reading and writing the whole n x l sketch per pivot.
//
// FP64 arithmetic issues one warp instruction per ~70 cycles and SM quarter here, however few lanes
// of it are active, so it is kept out of the inner loops: sums of squares and the reflector's
// residual are carried as float-float pairs (products and sums by error-free transformations, 2^-46
// where what is subtracted from them, an FP32 coordinate, has 2^-24; the pivots and |R_mm| came out
// bit for bit those of FP64 sums on sketches of up to 10^5 x 1050), and what is FP64 per row (the
// downdated norm, the pivot key) is done for up to 32 rows of a warp at once, a lane each.  At
// n = 10^5, l = 1050, k = 1000, with FP64 sums and a warp's lane 0 for a row -> so:
//     norms      600 ->  92 us       reflector      19.3 -> 10.0 us a pivot
//     panel end  650 -> 150 us       pivot step     65   -> 53   us a pivot (5.3 TB/s and 15 us)
//     all of it  106 ->  70 ms
#include "internal.cuh"
#include "sym.cuh"

#include <algorithm>

namespace krr {

constexpr int QR_THREADS = 256;
constexpr int QR_WARPS = QR_THREADS / 32;
constexpr int QH_B = 32;   // pivots per panel
constexpr int QR_REF_THREADS = 1024;   // the one-block reflector kernel: short dependent chains
constexpr int QR_REF_WARPS = QR_REF_THREADS / 32;

// max key = largest residual norm, then lowest index
__device__ __forceinline__ unsigned long long pivot_key(double nrm2, long long i) {
    const float f = (float)fmax(nrm2, 0.0);
    return ((unsigned long long)__float_as_uint(f) << 32) | (unsigned long long)(0xffffffffu - (unsigned)i);
}
__device__ __forceinline__ long long key_index(unsigned long long k) {
    return (long long)(0xffffffffu - (unsigned)(k & 0xffffffffu));
}

constexpr int QR_STEP_BLOCKS = 3;   // blocks of a pivot step on an SM at most
constexpr int QR_RB = 8;      // rows of a warp whose norms are taken together

// (h, l) += x * y exactly to the pair's precision
__device__ __forceinline__ void qr_ff_mad(float& h, float& l, float x, float y) {
    const float p = __fmul_rn(x, y), pe = fmaf(x, y, -p);
    const float s = __fadd_rn(h, p), z = __fsub_rn(s, h);
    const float e = __fadd_rn(__fsub_rn(h, __fsub_rn(s, z)), __fsub_rn(p, z));
    h = s;
    l = __fadd_rn(l, __fadd_rn(e, pe));
}
// a sum of squares the pair holds: below, the products' low parts underflow; above (or not finite),
// products overflow.  Outside it the sums are taken again in FP64.
__device__ __forceinline__ bool qr_ff_range(float h) { return h > 1e-24f && h < 1e36f; }

// the pair summed over the warp, in every lane
__device__ __forceinline__ void qr_ff_warp(float& h, float& l) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const float oh = __shfl_xor_sync(0xffffffffu, h, o), ol = __shfl_xor_sync(0xffffffffu, l, o);
        const float s = __fadd_rn(h, oh), z = __fsub_rn(s, h);
        const float e = __fadd_rn(__fsub_rn(h, __fsub_rn(s, z)), __fsub_rn(oh, z));
        l = __fadd_rn(__fadd_rn(l, ol), e);
        h = s;
    }
}
// a row's sum of squares in FP64, by a warp
__device__ __forceinline__ double qr_sumsq64(const float* y, int L, int lane) {
    double s = 0.0;
    for (int t = lane; t < L; t += 32) s = fma((double)y[t], (double)y[t], s);
    return warp_sum(s);
}
// the pair normalised, its square added to (sh, sl)
__device__ __forceinline__ float2 qr_ff_norm(float h, float l, float& sh, float& sl) {
    const float z = __fadd_rn(h, l);
    l = __fsub_rn(l, __fsub_rn(z, h));
    qr_ff_mad(sh, sl, z, z);
    sl = fmaf(2.f * z, l, sl);
    return make_float2(z, l);
}
// coordinate t of the pivot row's residual in FP64
__device__ __forceinline__ double qr_z64(const float* yp, const float* cps, const float* Vp, int l, int jm, int t) {
    double z = yp[t];
    for (int j = 0; j < jm; ++j) z -= (double)cps[j] * (double)Vp[(size_t)j * l + t];
    return z;
}

// the block's best key into bkeys[blockIdx.x]
template <int WARPS>
__device__ __forceinline__ void qr_block_key(unsigned long long best, unsigned long long* bkeys) {
    __shared__ unsigned long long sbest[WARPS];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) best = max(best, __shfl_xor_sync(0xffffffffu, best, o));
    if ((threadIdx.x & 31) == 0) sbest[threadIdx.x >> 5] = best;
    __syncthreads();
    if (threadIdx.x == 0) {
        unsigned long long b = 0;
        for (int w = 0; w < WARPS; ++w) b = max(b, sbest[w]);
        bkeys[blockIdx.x] = b;   // reduced by the next reflector (no atomic contention)
    }
}

// residual norms of all rows and the key of the first pivot
__global__ void __launch_bounds__(QR_THREADS)
k_qr_norms(const float* __restrict__ Y, long long n, int l, int ldy, double* __restrict__ nrm,
           unsigned long long* __restrict__ bkeys) {
    pdl_entry();
    const int lane = threadIdx.x & 31;
    const long long w0 = (long long)blockIdx.x * QR_WARPS + (threadIdx.x >> 5);
    const long long nw = (long long)gridDim.x * QR_WARPS;
    unsigned long long best = 0;
    for (long long i0 = w0 * QR_RB; i0 < n; i0 += nw * QR_RB) {
        float mh = 0.f, ml = 0.f;                  // lane r < QR_RB: row i0 + r
        double s64 = -1.0;
        for (int r = 0; r < QR_RB && i0 + r < n; ++r) {
            float h = 0.f, l2 = 0.f;
            for (int c = lane; c < l; c += 32) {
                const float v = Y[(i0 + r) * ldy + c];
                qr_ff_mad(h, l2, v, v);
            }
            qr_ff_warp(h, l2);
            if (lane == r) mh = h, ml = l2;
            if (!qr_ff_range(h)) {
                const double s = qr_sumsq64(Y + (i0 + r) * ldy, l, lane);
                if (lane == r) s64 = s;
            }
        }
        if (lane < QR_RB && i0 + lane < n) {
            const double s = s64 >= 0.0 ? s64 : (double)mh + (double)ml;
            nrm[i0 + lane] = s;
            best = max(best, pivot_key(s, i0 + lane));
        }
    }
    qr_block_key<QR_WARPS>(best, bkeys);
}

// Reflector of pivot step m (panel column jm = m - m0), one block: the pivot row's
// residual z = y_p^(m0)[m:] - sum_{j<jm} c[p][j] v_j[m:], then v = z / (z_0 - alpha) with
// alpha = -sign(z_0) ||z||, tau = (alpha - z_0) / alpha (v_0 = 1), and g_j = v . v_j[m:]
// for the earlier reflectors of the panel.  Writes the pivot, |R_mm| = ||z|| and marks
// the row chosen.  A chain of latencies: the panel's reflectors do not depend on the pivot, so a
// thread's first coordinate of all of them is loaded (into registers, used for z and for g) before
// the pivot is known.
__global__ void __launch_bounds__(QR_REF_THREADS, 1)
k_qr_reflector(const float* __restrict__ Y, long long n, int l, int ldy, int m, int jm, const float* __restrict__ C,
               float* __restrict__ Vp, float* __restrict__ tau, float* __restrict__ g,
               double* __restrict__ nrm, const unsigned long long* __restrict__ bkeys, int nbk,
               int* __restrict__ piv, float* __restrict__ rdiag, const int* __restrict__ forced,
               float* __restrict__ Rout) {
    pdl_entry();
    extern __shared__ float2 zs[];   // z in pairs, by coordinate
    __shared__ double red[QR_REF_WARPS];
    __shared__ float2 redf[QR_REF_WARPS];
    __shared__ unsigned long long kred[QR_REF_WARPS];
    __shared__ double s_scale;
    __shared__ int s_redo;
    __shared__ float cps[QH_B];
    __shared__ float gred[QR_REF_WARPS][QH_B];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = blockDim.x >> 5;
    const int t0 = threadIdx.x;      // this thread's first coordinate
    float vj[QH_B];
#pragma unroll
    for (int j = 0; j < QH_B; ++j) vj[j] = j < jm && t0 >= m && t0 < l ? Vp[(size_t)j * l + t0] : 0.f;
    // the pivot: the largest of the previous pass's per-block keys
    {
        unsigned long long b = 0;
        for (int i = threadIdx.x; i < nbk; i += blockDim.x) b = max(b, bkeys[i]);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) b = max(b, __shfl_xor_sync(0xffffffffu, b, o));
        if (lane == 0) kred[w] = b;
        __syncthreads();
    }
    unsigned long long km = lane < nw ? kred[lane] : 0ull;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) km = max(km, __shfl_xor_sync(0xffffffffu, km, o));
    // the argmax, or the caller's pivot (strong RRQR re-factorizes with a given order)
    if (forced) km = 1ull;
    const long long p = forced ? (long long)forced[m] : key_index(km);
    if (km == 0 || p < 0 || p >= n) {   // no candidate left (cannot happen for k <= n): stop
        if (threadIdx.x == 0) {
            piv[m] = 0;
            rdiag[m] = 0.f;
            tau[jm] = 0.f;
        }
        for (int t = threadIdx.x; t < l; t += blockDim.x) Vp[(size_t)jm * l + t] = 0.f;
        if (threadIdx.x < jm) g[threadIdx.x] = 0.f;
        return;
    }
    const float* yp = Y + p * ldy;
    const float* cp = C + p * QH_B;
    const float y0 = t0 >= m && t0 < l ? yp[t0] : 0.f;
    if (threadIdx.x < QH_B) cps[threadIdx.x] = threadIdx.x < jm ? cp[threadIdx.x] : 0.f;
    __syncthreads();
    float sh = 0.f, sl = 0.f;                      // sum of squares
    if (t0 >= m && t0 < l) {
        float h = y0, lo = 0.f;
#pragma unroll
        for (int j = 0; j < QH_B; ++j)
            if (j < jm) qr_ff_mad(h, lo, -cps[j], vj[j]);
        zs[t0] = qr_ff_norm(h, lo, sh, sl);
    }
    for (int t = t0 + blockDim.x; t < l; t += blockDim.x) {
        if (t < m) continue;
        float h = yp[t], lo = 0.f;
#pragma unroll 4
        for (int j = 0; j < jm; ++j) qr_ff_mad(h, lo, -cps[j], Vp[(size_t)j * l + t]);
        zs[t] = qr_ff_norm(h, lo, sh, sl);
    }
    __syncwarp();
    qr_ff_warp(sh, sl);
    if (lane == 0) redf[w] = make_float2(sh, sl);
    __syncthreads();
    double z0 = 0.0, t2 = 0.0;
    if (w == 0) {
        const float2 f = lane < nw ? redf[lane] : make_float2(0.f, 0.f);
        float h = f.x, lo = f.y;
        qr_ff_warp(h, lo);
        if (lane == 0) s_redo = !qr_ff_range(h);
        z0 = (double)zs[m].x + (double)zs[m].y;
        t2 = (double)h + (double)lo;
    }
    __syncthreads();
    const bool redo = s_redo != 0;
    if (redo) {   // squares outside the pair's range: z and its norm in FP64
        double ss = 0.0;
        for (int t = t0; t < l; t += blockDim.x) {
            if (t < m) continue;
            const double z = qr_z64(yp, cps, Vp, l, jm, t);
            ss = fma(z, z, ss);
        }
        __syncwarp();
        ss = warp_sum(ss);
        if (lane == 0) red[w] = ss;
        __syncthreads();
        if (w == 0) {
            z0 = qr_z64(yp, cps, Vp, l, jm, m);
            t2 = warp_sum(lane < nw ? red[lane] : 0.0);
        }
    }
    if (w == 0) {                                  // both quotients at once, a lane each
        const double nz = sqrt(t2);
        const double alpha = z0 >= 0.0 ? -nz : nz;
        const bool on = nz > 0.0 && z0 - alpha != 0.0;
        const double num = lane == 0 ? 1.0 : alpha - z0, den = lane == 0 ? z0 - alpha : alpha;
        const double q = on ? num / den : 0.0;
        if (lane == 0) {
            s_scale = q;
            piv[m] = (int)p;
            rdiag[m] = (float)nz;
            nrm[p] = -1.0;
            if (Rout) Rout[(size_t)m * n + p] = (float)alpha;   // R_mm
        }
        if (lane == 1) tau[jm] = (float)q;
    }
    __syncthreads();
    float* vm = Vp + (size_t)jm * l;
    const double scale = s_scale;
    // g_j = v . v_j[m:] for j < jm: every thread sums its coordinates for all j at once, in place
    // of the reflectors' values, then the lanes and the warps in order
    auto v_of = [&](int t) {
        if (t <= m) return t == m ? 1.f : 0.f;
        const double z = redo ? qr_z64(yp, cps, Vp, l, jm, t) : (double)zs[t].x + (double)zs[t].y;
        return (float)(z * scale);
    };
    if (t0 < l) {
        const float v = v_of(t0);
        vm[t0] = v;
#pragma unroll
        for (int j = 0; j < QH_B; ++j) vj[j] *= v;
    }
#pragma unroll 1
    for (int t = t0 + blockDim.x; t < l; t += blockDim.x) {
        const float v = v_of(t);
        vm[t] = v;
        if (t < m) continue;
#pragma unroll
        for (int j = 0; j < QH_B; ++j)
            if (j < jm) vj[j] = fmaf(v, Vp[(size_t)j * l + t], vj[j]);
    }
    __syncwarp();
    lane_sum<QH_B, 16>(vj, lane);                  // lane j: the warp's g_j
    gred[w][lane] = vj[0];
    __syncthreads();
    if (threadIdx.x < jm) {
        float gs = 0.f;
#pragma unroll 8
        for (int i = 0; i < nw; ++i) gs += gred[i][threadIdx.x];
        g[threadIdx.x] = gs;
    }
}

__device__ __forceinline__ void qr_cp4(float* dst, const float* src) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src)
                 : "memory");
}

// Pivot step m: for every row not chosen, c[i][jm] = tau (v . y_i^(m0)[m:] - sum_j c[i][j] g_j),
// its coordinate r = y_i^(m0)[m] - sum_j c[i][j] v_j[m] - c[i][jm], and nrm_i -= r^2; the
// key of the next pivot.  Bound by reading the rows' coordinates m..l-1.  A warp takes rw rows (a
// multiple of U), U at a time, copied asynchronously into its own ring of D shared buffers (kp
// 32-wide pieces a row, whatever their alignment, then the row's c): about 4 KB a buffer keeps the
// reads in flight without holding registers.  A lane reads only what it copied.  The three sums and
// the first coordinate of the U rows are reduced over the lanes together and handed to the rows'
// lanes, which do the FP64 work of 32 rows at a time.
template <int U, int D>
__global__ void __launch_bounds__(QR_THREADS)
k_qr_step(const float* __restrict__ Y, long long n, int l, int ldy, int m, int jm, int rw, int kp,
          float* __restrict__ C, const float* __restrict__ Vp, const float* __restrict__ tau,
          const float* __restrict__ g, double* __restrict__ nrm, unsigned long long* __restrict__ bkeys,
          float* __restrict__ Rout) {
    pdl_entry();
    constexpr int S = U == 8 ? 0 : U == 4 ? 1 : U == 2 ? 2 : 3;   // value q of row u: in lane (4 u + q) 2^S
    extern __shared__ float qsm[];    // v_m[m:] zero-padded, then the warps' rings
    __shared__ float gsh[QH_B], vjm[QH_B];
    const int L = l - m, row = 32 * (kp + 1);
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    float* ring = qsm + 32 * kp + wid * (D * U) * row + lane;
    const float* vm = Vp + (size_t)jm * l + m;
    for (int t = threadIdx.x; t < kp * 32; t += QR_THREADS) qsm[t] = t < L ? vm[t] : 0.f;
    if (threadIdx.x < QH_B) {
        gsh[threadIdx.x] = threadIdx.x < jm ? g[threadIdx.x] : 0.f;
        vjm[threadIdx.x] = threadIdx.x < jm ? Vp[(size_t)threadIdx.x * l + m] : 0.f;
    }
    // what the copies leave out: the last piece beyond the row's end, and c from jm on
    const bool tail = lane + 32 * (kp - 1) < L, cin = lane < jm;
    for (int b = 0; b < D * U; ++b) {
        if (!tail) ring[b * row + 32 * (kp - 1)] = 0.f;
        if (!cin) ring[b * row + 32 * kp] = 0.f;
    }
    __syncthreads();
    const float tu = tau[jm];
    const float gl = gsh[lane], vl = vjm[lane];
    const long long first = ((long long)blockIdx.x * QR_WARPS + wid) * rw;
    const long long last = min(n, first + rw);
    long long ci = first;                          // the next U rows to copy
    int cslot = 0;
    auto copy = [&]() {
        if (ci < last) {
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const long long i = min(ci + u, n - 1);
                const float* src = Y + i * ldy + m + lane;
                float* dst = ring + (cslot * U + u) * row;
                for (int k = 0; k < kp - 1; ++k) qr_cp4(dst + 32 * k, src + 32 * k);
                if (tail) qr_cp4(dst + 32 * (kp - 1), src + 32 * (kp - 1));
                if (cin) qr_cp4(dst + 32 * kp, C + i * QH_B + lane);
            }
            ci += U;
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
        cslot = cslot + 1 == D ? 0 : cslot + 1;
    };
#pragma unroll
    for (int s = 0; s < D - 1; ++s) copy();
    unsigned long long best = 0;
    int slot = 0;
    for (long long i0 = first; i0 < last; i0 += 32) {
        const long long mine = i0 + lane;          // the row whose FP64 work this lane does
        const bool on = mine < last;
        const double ni = on ? nrm[mine] : -1.0;
        float dot = 0.f, corr = 0.f, shift = 0.f, y0 = 0.f;
#pragma unroll 1
        for (int r0 = 0; r0 < 32 && i0 + r0 < last; r0 += U) {
            copy();
            asm volatile("cp.async.wait_group %0;" ::"n"(D - 1) : "memory");
            const float* ys = ring + slot * U * row;
            float a[4 * U];
#pragma unroll
            for (int u = 0; u < U; ++u) a[4 * u] = 0.f;
#pragma unroll 4
            for (int k = 0; k < kp; ++k) {
                const float v = qsm[lane + 32 * k];
#pragma unroll
                for (int u = 0; u < U; ++u) a[4 * u] = fmaf(ys[u * row + 32 * k], v, a[4 * u]);
            }
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const float c = ys[u * row + 32 * kp];
                a[4 * u + 1] = c * gl;
                a[4 * u + 2] = c * vl;
                a[4 * u + 3] = lane == 0 ? ys[u * row] : 0.f;
            }
            lane_sum<4 * U, 16>(a, lane);
#pragma unroll
            for (int o = (1 << S) / 2; o >= 1; o >>= 1) a[0] += __shfl_xor_sync(0xffffffffu, a[0], o);
            const int src = (4 * (lane - r0)) << S;
            const float a0 = __shfl_sync(0xffffffffu, a[0], src);
            const float a1 = __shfl_sync(0xffffffffu, a[0], src + (1 << S));
            const float a2 = __shfl_sync(0xffffffffu, a[0], src + (2 << S));
            const float a3 = __shfl_sync(0xffffffffu, a[0], src + (3 << S));
            if (lane >= r0 && lane < r0 + U) dot = a0, corr = a1, shift = a2, y0 = a3;
            slot = slot + 1 == D ? 0 : slot + 1;
        }
        if (on && !(ni < 0.0)) {                   // not chosen
            const float cm = tu * (dot - corr);
            C[mine * QH_B + jm] = cm;
            const double r = (double)y0 - (double)shift - (double)cm;
            if (Rout) Rout[(size_t)m * n + mine] = (float)r;   // R_mi: coordinate m of row i
            const double nn = fmax(ni - r * r, 0.0);
            nrm[mine] = nn;
            best = max(best, pivot_key(nn, mine));
        }
    }
    asm volatile("cp.async.wait_all;" ::: "memory");
    qr_block_key<QR_WARPS>(best, bkeys);
}

typedef void (*qr_step_fn)(const float*, long long, int, int, int, int, int, int, float*, const float*, const float*,
                           const float*, double*, unsigned long long*, float*);
struct QrStep {
    qr_step_fn fn;
    int U, D;
};
// buffers of about 4 KB, as many as leave two blocks on an SM (kp <= 32)
static QrStep qr_step_for(int kp) {
    if (kp <= 4) return {&k_qr_step<8, 2>, 8, 2};
    if (kp <= 8) return {&k_qr_step<4, 3>, 4, 3};
    if (kp <= 16) return {&k_qr_step<2, 3>, 2, 3};
    if (kp <= 32) return {&k_qr_step<1, 3>, 1, 3};
    if (kp <= 64) return {&k_qr_step<1, 2>, 1, 2};
    return {&k_qr_step<1, 1>, 1, 1};
}

// Panel end (nb reflectors, coordinates m1..l-1 with m1 = m0 + nb): y_i[m1:] -= sum_j
// c[i][j] v_j[m1:] for the rows not chosen, then their residual norms afresh and
// the key of the next pivot.  The panel's reflectors are in shared memory (one block to an SM); a
// warp takes QP_R rows and QP_T 32-wide coordinate groups at a time, so that a reflector's value is
// read once for QP_R rows and a row's coefficient (broadcast) once for QP_T coordinates: with a row
// at a time the shared memory reads bound it, 650 us on average at n = 10^5, l = 1050.
constexpr int QP_THREADS = 512, QP_WARPS = QP_THREADS / 32;
constexpr int QP_R = 8, QP_T = 4;
__host__ __device__ inline size_t qp_smem(int nb, int L) {
    return sizeof(float) * ((size_t)QP_WARPS * QH_B * QP_R + (size_t)nb * L + 32 * QP_T);
}
__global__ void __launch_bounds__(QP_THREADS, 1)
k_qr_panel(float* __restrict__ Y, long long n, int l, int ldy, int m1, int nb, const float* __restrict__ C,
           const float* __restrict__ Vp, double* __restrict__ nrm, unsigned long long* __restrict__ bkeys) {
    pdl_entry();
    extern __shared__ __align__(16) float qps[];   // the warps' coefficients, then nb x L reflectors
    const int L = l - m1;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    float4* cs = reinterpret_cast<float4*>(qps + (size_t)wid * QH_B * QP_R);   // [j][row]
    float* vps = qps + (size_t)QP_WARPS * QH_B * QP_R;
    for (int j = wid; j < nb; j += QP_WARPS)
        for (int t = lane; t < L; t += 32) vps[j * L + t] = Vp[(size_t)j * l + m1 + t];
    if (threadIdx.x < 32 * QP_T) vps[nb * L + threadIdx.x] = 0.f;   // read past the last one's end
    __syncthreads();
    unsigned long long best = 0;
    // groups of rows dealt to the blocks first: few of them still reach every SM
    for (long long i0 = ((long long)wid * gridDim.x + blockIdx.x) * QP_R; i0 < n;
         i0 += (long long)QP_WARPS * gridDim.x * QP_R) {
        const bool on = lane < QP_R && i0 + lane < n;
        const unsigned left = __ballot_sync(0xffffffffu, on && !(nrm[i0 + lane] < 0.0));   // not chosen
        __syncwarp();
#pragma unroll
        for (int q = 0; q < QP_R / 4; ++q) {
            float c[4];
#pragma unroll
            for (int r = 0; r < 4; ++r) c[r] = -C[min(i0 + 4 * q + r, n - 1) * QH_B + lane];
            cs[lane * (QP_R / 4) + q] = make_float4(c[0], c[1], c[2], c[3]);
        }
        __syncwarp();
        float* yg = Y + i0 * ldy + m1;
        float h[QP_R], lo[QP_R];
#pragma unroll
        for (int r = 0; r < QP_R; ++r) h[r] = lo[r] = 0.f;
        for (int t0 = lane; t0 < L + lane; t0 += 32 * QP_T) {
            float y[QP_R][QP_T];
#pragma unroll
            for (int r = 0; r < QP_R; ++r)
#pragma unroll
                for (int u = 0; u < QP_T; ++u)
                    y[r][u] = ((left >> r) & 1u) && t0 + 32 * u < L ? yg[(size_t)r * ldy + t0 + 32 * u] : 0.f;
#pragma unroll 2
            for (int j = 0; j < nb; ++j) {
                const float4 ca = cs[2 * j], cb = cs[2 * j + 1];
                const float c[QP_R] = {ca.x, ca.y, ca.z, ca.w, cb.x, cb.y, cb.z, cb.w};
#pragma unroll
                for (int u = 0; u < QP_T; ++u) {
                    const float v = vps[j * L + t0 + 32 * u];
#pragma unroll
                    for (int r = 0; r < QP_R; ++r) y[r][u] = fmaf(c[r], v, y[r][u]);
                }
            }
#pragma unroll
            for (int r = 0; r < QP_R; ++r)
#pragma unroll
                for (int u = 0; u < QP_T; ++u)
                    if (((left >> r) & 1u) && t0 + 32 * u < L) {
                        yg[(size_t)r * ldy + t0 + 32 * u] = y[r][u];
                        qr_ff_mad(h[r], lo[r], y[r][u], y[r][u]);
                    }
        }
        float mh = 0.f, ml = 0.f;                  // lane r < QP_R: row i0 + r
        double s64 = -1.0;
#pragma unroll
        for (int r = 0; r < QP_R; ++r) {
            qr_ff_warp(h[r], lo[r]);
            if (lane == r) mh = h[r], ml = lo[r];
            if (((left >> r) & 1u) && !qr_ff_range(h[r])) {
                const double s = qr_sumsq64(yg + (size_t)r * ldy, L, lane);
                if (lane == r) s64 = s;
            }
        }
        if ((left >> lane) & 1u) {
            const double s = s64 >= 0.0 ? s64 : (double)mh + (double)ml;
            nrm[i0 + lane] = s;
            best = max(best, pivot_key(s, i0 + lane));
        }
    }
    qr_block_key<QP_WARPS>(best, bkeys);
}

// The pivoted QR of Y^T (Y n x ldy, l used columns) for k pivots.  forced (device, k) makes
// step m take pivot forced[m] instead of the argmax; Rout (device, k x n) receives row m of R
// for every column (the pivot's diagonal, the rows not yet chosen; chosen ones are left
// alone), and then the last step runs too, so that nrm ends as the squared residual norms
// after k pivots (-1 for the chosen rows).
int qrcp_core(krr_ctx* ctx, float* Y, long long n, int l, int ldy, int k, int* piv, float* rdiag,
              const int* forced, float* Rout, double** nrm_out) {
    if (l > 4096) return fail(ctx, KRR_E_INVAL, "qrcp: more than 4096 projections");
    if (n >= 0xffffffffLL) return fail(ctx, KRR_E_INVAL, "qrcp: too many points");
    if (k > l) return fail(ctx, KRR_E_INVAL, "qrcp: more pivots than projections");
    // enough warps for every row's loads to be in flight within a few waves; every pass
    // writes one key per block, which the next reflector reduces
    const int grid = (int)std::min<long long>((long long)ctx->num_sms * 8, ceil_div(n, QR_WARPS * QR_RB));
    double* nrm;
    float *C, *Vp, *tau, *g;
    unsigned long long* bkeys;
    KRR_RET(bufT(ctx, "qr_nrm64", (size_t)n, &nrm));
    KRR_RET(bufT(ctx, "qr_c", (size_t)n * QH_B, &C));
    KRR_RET(bufT(ctx, "qr_v", (size_t)QH_B * l, &Vp));
    KRR_RET(bufT(ctx, "qr_tau", (size_t)QH_B, &tau));
    KRR_RET(bufT(ctx, "qr_g", (size_t)QH_B, &g));
    KRR_RET(bufT(ctx, "qr_bkeys", (size_t)std::max(grid, ctx->num_sms * QR_STEP_BLOCKS), &bkeys));
    KRR_RET(allow_max_dynamic_smem(ctx, (const void*)k_qr_panel));
    // panel width: the panel's reflectors (nb x l floats) must fit 200 KB of shared memory
    const int ref_threads = std::min(QR_REF_THREADS, (int)ceil_div(l, 32) * 32);
    const int bmax = std::max(1, std::min(QH_B, (200 * 1024) / (4 * l)));
    k_qr_norms<<<grid, QR_THREADS, 0, ctx->stream>>>(Y, n, l, ldy, nrm, bkeys);
    KRR_CHECK_LAUNCH();
    int nbk = grid;   // keys of the last pass
    for (int m0 = 0; m0 < k; m0 += bmax) {
        const int nb = std::min(bmax, k - m0);
        for (int jm = 0; jm < nb; ++jm) {
            const int m = m0 + jm;
            const int L = l - m;
            launch_pdl(k_qr_reflector, 1, ref_threads, sizeof(float2) * l, ctx->stream, Y, n, l, ldy, m, jm, C, Vp,
                       tau, g, nrm, bkeys, nbk, piv, rdiag, forced, Rout);
            KRR_CHECK_LAUNCH();
            if (m + 1 < k || Rout) {
                const int kp = (L + 31) / 32;
                const QrStep st = qr_step_for(kp);
                const size_t smem = 4 * 32 * ((size_t)kp + (size_t)QR_WARPS * st.U * st.D * (kp + 1));
                KRR_RET(allow_max_dynamic_smem(ctx, (const void*)st.fn));
                // equal runs of rows for the warps that are resident together
                const int per_sm = std::max(1, std::min(QR_STEP_BLOCKS, (int)(220 * 1024 / smem)));
                const int rw = (int)ceil_div(n, (long long)ctx->num_sms * per_sm * QR_WARPS * st.U) * st.U;
                nbk = (int)ceil_div(n, (long long)QR_WARPS * rw);
                launch_pdl(st.fn, nbk, QR_THREADS, smem, ctx->stream, Y, n, l, ldy, m, jm, rw, kp, C, Vp, tau, g,
                           nrm, bkeys, Rout);
                KRR_CHECK_LAUNCH();
            }
        }
        const int m1 = m0 + nb;
        if (m1 < k) {
            // the panel's updates reach the coordinates beyond it; the exact norms replace
            // the downdated ones and give the next pivot
            nbk = (int)std::min<long long>(ctx->num_sms, ceil_div(n, QP_R));
            launch_pdl(k_qr_panel, nbk, QP_THREADS, qp_smem(nb, l - m1), ctx->stream, Y, n, l, ldy, m1, nb, C, Vp,
                       nrm, bkeys);
            KRR_CHECK_LAUNCH();
        }
    }
    if (nrm_out) *nrm_out = nrm;
    return KRR_OK;
}

int launch_qrcp(krr_ctx* ctx, float* Y, long long n, int l, int ldy, int k, int* piv, float* rdiag) {
    return qrcp_core(ctx, Y, n, l, ldy, k, piv, rdiag, nullptr, nullptr, nullptr);
}

}  // namespace krr

// Shared by the symmetric products (sym_tc.cu, sym_f32.cu): the order and split of their work, the
// layout of their partial sums, and lane reductions.
#pragma once

#include "internal.cuh"

namespace krr {

constexpr int SY_T = 128;                        // rows per tile

// The points in column units of BN and row blocks of RU units (RU * BN / 128 row tiles).  Row
// block I has the units I * RU .. NU - 1; first(I) (block, unit) pairs come before its own.
struct SyGrid {
    int n, BN, NU, RU, nblk, G;
    long long W;                                  // (block, unit) pairs in all
    __host__ __device__ int row_tiles(int I) const { return min(RU, NU - I * RU) * (BN / SY_T); }
    __host__ __device__ int rows() const { return RU * BN; }
    __host__ __device__ long long first(int I) const {
        return (long long)I * NU - (long long)RU * ((long long)I * (I - 1) / 2);
    }
    // the row block of pair u
    __host__ __device__ int block_of(long long u) const {
        int lo = 0, hi = nblk - 1;
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (first(mid) <= u) lo = mid;
            else hi = mid - 1;
        }
        return lo;
    }
    __host__ __device__ long long run_begin(int s) const { return W * s / G; }
    // the run that holds pair u: the largest s with run_begin(s) <= u
    __host__ __device__ int run_of(long long u) const { return (int)(((u + 1) * G - 1) / W); }
    // first entry of column unit T's slots (T / RU of them, BN entries each)
    __host__ __device__ long long col_base(int T) const {
        const long long b = T / RU, r = T % RU;
        return BN * (RU * (b * (b - 1) / 2) + r * b);
    }
    // the slot of row block I, and the slots of a column unit of block b
    __host__ __device__ int slot(int I) const { return I; }
    __host__ __device__ int slots(int b) const { return b; }
    __host__ __device__ bool first_panel() const { return true; }
    __host__ __device__ bool last_panel() const { return true; }
    __host__ __device__ bool has(int) const { return true; }
    static __host__ __device__ int min(int a, int b) { return a < b ? a : b; }
};

// Most bytes of column sums that a context holds for the products of one point set.  Without a limit
// they grew as 4 n^2 / rows() (4 GB at n = 10^6 with 1024-row blocks, 16 GB with 256).  256 MB are the
// sums of 2.6 10^5 points on the tensor cores with 64-wide features, of 1.8 10^5 with 128-wide ones and
// of 1.3 10^5 in FP32; larger sets take the row blocks in panels, a launch and a reduction each.
// d = 8, in panels and with all sums (0.6 GB) held: FP32, n = 2 10^5 9.97 and 9.70 ms; tensor cores,
// n = 4 10^5 14.2 and 14.4 ms.
constexpr long long kSymBytes = 256LL << 20;

// The row blocks I0 .. I1 - 1 of a grid, whose W pairs from number u0 on are cut into G runs.  A type of
// its own, for which the kernels are compiled again: the plain one's addresses stay as short as they are.
struct SyPanel : SyGrid {
    int I0, I1;
    long long u0;
    __host__ __device__ long long run_begin(int s) const { return u0 + W * s / G; }
    __host__ __device__ int run_of(long long u) const { return (int)(((u - u0 + 1) * G - 1) / W); }
    __host__ __device__ int slot(int I) const { return I - I0; }
    __host__ __device__ int slots(int b) const { return b <= I0 ? 0 : min(b, I1) - I0; }
    __host__ __device__ long long col_base(int T) const {
        const long long m = slots(T / RU), units = T - (I0 + m) * RU;   // units with m slots before T
        return m == 0 ? 0 : BN * (RU * (m * (m - 1) / 2) + units * m);
    }
    __host__ __device__ bool first_panel() const { return I0 == 0; }
    __host__ __device__ bool last_panel() const { return I1 == nblk; }
    __host__ __device__ bool has(int b) const { return b >= I0 && b < I1; }
    long long col_entries() const {
        const long long m = I1 - I0, beyond = NU - (long long)I1 * RU;
        return BN * (RU * (m * (m - 1) / 2) + (beyond > 0 ? beyond : 0) * m);
    }
    // The panel from row block I on: as many blocks as `entries` column sums hold, one at least, in up to
    // maxruns runs.
    SyPanel(const SyGrid& g, int I, long long entries, int maxruns) : SyGrid(g), I0(I) {
        int lo = I0 + 1, hi = nblk;                // the entries grow with the blocks
        while (lo < hi) {
            I1 = lo + (hi - lo + 1) / 2;
            if (col_entries() <= entries) lo = I1;
            else hi = I1 - 1;
        }
        I1 = lo;
        u0 = first(I0);
        W = first(I1) - u0;
        G = (int)(W < maxruns ? W : maxruns);
    }
};

// Sums each a[m] over the lanes that differ in bit ST and the lower bits halved in turn, down to
// N >> levels values: a lane keeps the half of the values its bit selects and sends the other.
template <int N, int ST, class T>
__device__ __forceinline__ void lane_sum(T* a, int lane) {
    constexpr int H = N / 2;
    const bool up = (lane & ST) != 0;
#pragma unroll
    for (int m = 0; m < H; ++m) {
        const T send = up ? a[m] : a[m + H];
        const T keep = up ? a[m + H] : a[m];
        a[m] = keep + __shfl_xor_sync(0xffffffffu, send, ST);
    }
    if constexpr (H > 1) lane_sum<H, ST / 2>(a, lane);
}

__device__ __forceinline__ unsigned long long sy_pack(float lo, float hi) {
    unsigned long long r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
    return r;
}
__device__ __forceinline__ void sy_unpack(unsigned long long v, float& lo, float& hi) {
    asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v));
}
__device__ __forceinline__ void sy_fma(unsigned long long& d, unsigned long long a, unsigned long long b) {
    asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(d) : "l"(a), "l"(b));
}

// The points of an FP32 product as its kernel has them (packed, or raw coordinates with nsc != 0), for
// the sums that leave the range of its float pairs; P null where v was scaled so that none does.
struct SyPoints {
    const float* P = nullptr;
    int d = 0, ps = 0;
    float nsc = 0.f;
};

// The two buffers of partial sums of a product of up to G runs, shared by all forms (8 bytes an entry).
// KRR_E_NOMEM where they do not fit the device, without another try while krr_ctx::sym_nomem says so.
int sym_buffers(krr_ctx* ctx, const SyGrid& g, void** row, void** col);

// Q = ksc vscale (row and column partial sums) + beta V (vscale: device, null for 1), or with a panel that
// is not the last the running sums.  Defined in sym_tc.cu for SyGrid and SyPanel.
template <class Grid>
int launch_sym_reduce(krr_ctx* ctx, const Grid& g, const float2* rowpart, const float2* colpart, const float* V,
                      float beta, double ksc, const double* vscale, float* Q, SyPoints pts);

// One product in all of its launches: f(grid, rowpart, colpart) for the grid as it is or for each panel,
// on the buffers that all of them share.
template <class F>
inline int sym_product(krr_ctx* ctx, const SyGrid& g, F&& f) {
    void *row, *col;
    KRR_RET(sym_buffers(ctx, g, &row, &col));
    if (8 * g.col_base(g.NU) <= kSymBytes) return f(g, row, col);
    for (int I = 0; I < g.nblk;) {
        const SyPanel p(g, I, kSymBytes / 8, g.G);
        KRR_RET(f(p, row, col));
        I = p.I1;
    }
    return KRR_OK;
}

}  // namespace krr

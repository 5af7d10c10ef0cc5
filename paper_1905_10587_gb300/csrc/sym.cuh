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
    static __host__ __device__ int min(int a, int b) { return a < b ? a : b; }
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

// Q = ksc vscale (row and column partial sums) + beta V (vscale: device, null for 1)
int launch_sym_reduce(krr_ctx* ctx, const SyGrid& g, const float2* rowpart, const float2* colpart, const float* V,
                      float beta, double ksc, const double* vscale, float* Q, SyPoints pts = SyPoints());

}  // namespace krr

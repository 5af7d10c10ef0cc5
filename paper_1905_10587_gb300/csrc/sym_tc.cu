// Symmetric tensor-core product: Q = (K(X, X) + beta I) v for one right-hand side, with every
// kernel value of a pair i < j evaluated once and used for both q_i and q_j.
//
// What bounds it: one ex2 (MUFU, 32 per SM and clock) per evaluated entry.  k_kmvm_tc evaluates
// all n^2 entries; here an entry off the diagonal blocks serves two of them, which halves the
// exponentials, the exponent MMAs and the TMEM reads, for one more FMA per entry.
//
// Layout.  The points are in row tiles of 128 and column units of BN = 256 (128 with 128-wide
// features); a row block is up to 8 row tiles.  A unit of work is (row block I, column unit c at
// or right of the block): for every row tile r of I one tcgen05 product S = FA(r) . FB(c)^T gives
// 128 x BN exponents in TMEM, which eight epilogue warps (2 column halves x 4 TMEM lane quarters)
// read with tcgen05.ld.16x256b.  That shape leaves a thread with 4 rows x 8 columns of each 32 x 32
// block (a fragment layout), so that both sums stay short:
//   row sums     4 per tile and thread, 3 shuffles over the four threads that share the rows,
//                folded float-float into shared memory per row
//   column sums  BN / 8 accumulators a thread, kept in registers over the unit's row tiles;
//                7 shuffles per 32 columns over the eight row groups once per unit
// (32x32b loads leave one row x 32 columns a thread: 31 shuffles per 32 columns, 1.45 ms for the
// whole call below.)  The row block's feature tiles stay in shared memory over all its column units:
// 32 KB of column features a unit from L2, where streaming the row tiles past each unit would take
// 32 bytes per SM and clock.  Inside the diagonal block (column units of I itself) both triangles
// are evaluated and only the row sums are used.
//
// Split.  The (block, unit) pairs of all row blocks form one sequence, cut into one equal run per
// SM: no tail wave, and a run touches few row blocks.  Column sums leave as float-float pairs in
// slot I of their column unit, row sums in one slot per (run, row block); k_sym_reduce adds the
// slots of every point in a fixed order, so results do not depend on timing.  Large sets take their row
// blocks in panels (SyPanel), a launch each.
//
// Measured, n = 10^5, d = 8, the whole krr_kmvm call (about 0.09 ms of it packs points and features and
// adds the slots): 1.00 ms; 1.149 against 1.754 ms for k_kmvm_tc when both still took 0.21 ms to pack,
// n = 2048 0.114 against 0.131 ms then, and ahead at every n down to 200, so it takes every square
// product with one right-hand side.  The kernel keeps the MUFU 53 to 55% busy and issues in 56% of the
// cycles; the largest stall is fixed-latency dependences, with two warps per scheduler (437
// instructions per warp and tile, of which 256 are ex2 and FMA).  Sixteen epilogue warps (64 columns each) measured 5% slower, two warp groups on alternate
// tiles 10% slower.  Fetching v a tile ahead and asking for the next tile's barrier a step ahead
// gave 5% together, folding row and column sums under the next tile's exponentials 4%.
#include "internal.cuh"
#include "cg_scalar.cuh"
#include "sym.cuh"
#include "tc_ptx.cuh"

#include <algorithm>
#include <type_traits>

namespace krr {

constexpr int SY_EW = 8;                         // epilogue warps: 2 column halves x 4 lane quarters
constexpr int SY_THREADS = 32 * (2 + SY_EW);
constexpr int SY_RTMAX = 8;                      // most row tiles per block
// buffers of the quarters' column sums, by column unit width (see column_done)
constexpr int sy_nc(int BN) { return BN == 256 ? 3 : 4; }

struct SyShared {
    uint64_t a_full[SY_RTMAX], a_empty[SY_RTMAX], b_full[2], b_empty[2], t_full[4], t_empty[4],
        c_full[2][4], drain;
    uint32_t tbase;
    int abort;
};

__device__ __forceinline__ void sy_bar(int id, int threads) {
    asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(threads) : "memory");
}

// v zero-padded to whole tiles (16-byte aligned bulk copies; padding columns add nothing), and
// the largest |v| of every SY_PAD entries.
constexpr int SY_PAD = 1024;
__global__ void __launch_bounds__(SY_PAD) k_sym_pad(const float* __restrict__ V, int n, int np,
                                                    float* __restrict__ Vp, float* __restrict__ bmax) {
    pdl_entry();
    __shared__ float red[SY_PAD / 32];
    const int i = blockIdx.x * SY_PAD + threadIdx.x;
    const float v = i < n ? V[i] : 0.f;
    if (i < np) Vp[i] = v;
    const float m = warp_max(fabsf(v));
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = m;
    __syncthreads();
    if (threadIdx.x < 32) {
        const float x = warp_max(red[threadIdx.x]);
        if (threadIdx.x == 0) bmax[blockIdx.x] = x;
    }
}

// Roles: warp 0 copies, warp 1 issues MMAs, warps 2..9 are the epilogue.  Barriers:
//   a_full[r] / a_empty[r]   row tile r of the current row block
//   b_full[s] / b_empty[s]   column unit stage s: features and v (empty needs the MMAs and the
//                            8 warps' reads of v)
//   t_full[b] / t_empty[b]   TMEM buffer b (512 / BN of them)
//   c_full[g][i]             column half g's four column sums in buffer i
// Every wait is bounded.  A warp whose wait ran out sets the abort and error words and goes on
// without waiting, so that the block barriers below still match.
template <int NK, int BN, class Grid>
__global__ void __launch_bounds__(SY_THREADS, 1)
k_kmvm_sym(const unsigned char* __restrict__ FA, const unsigned char* __restrict__ FB, int Kp, Grid sg,
           const float* __restrict__ Vp, float2* __restrict__ rowpart, float2* __restrict__ colpart,
           const float* __restrict__ bmax, int nbmax, double* __restrict__ vscale, int* __restrict__ err,
           long long wlimit, int stall_copies, uint32_t korder) {
    pdl_entry();
    constexpr int NBUF = 512 / BN;                     // TMEM buffers
    constexpr int CT = BN / SY_T;                      // feature tiles per column unit
    constexpr int CW = BN / 2;                         // columns per epilogue warp
    constexpr int NC = sy_nc(BN);
    constexpr int NQ = CW / 32;                        // 32-column chunks of a warp
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    unsigned char* smem = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);
    const uint32_t tileF = 128u * Kp * 2u;             // bytes of one feature tile
    const int R = sg.rows();                           // rows per block
    unsigned char* sA = smem;                          // the block's row tiles
    unsigned char* sB = sA + (size_t)(R / SY_T) * tileF;            // 2 column units
    float* sV = reinterpret_cast<float*>(sB + 2u * CT * tileF);     // 2 x BN
    float2* sRow = reinterpret_cast<float2*>(sV + 2 * BN);          // 2 column halves x R
    float* sCol = reinterpret_cast<float*>(sRow + 2 * R);           // NC x 4 quarters x BN
    SyShared* sh = reinterpret_cast<SyShared*>(sCol + NC * 4 * BN);

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    if (tid == 0) {
        for (int r = 0; r < SY_RTMAX; ++r) {
            mbar_init(&sh->a_full[r], 1);
            mbar_init(&sh->a_empty[r], 1);
        }
        for (int s = 0; s < 2; ++s) {
            mbar_init(&sh->b_full[s], 1);
            mbar_init(&sh->b_empty[s], 1 + SY_EW);
        }
        for (int b = 0; b < NBUF; ++b) {
            mbar_init(&sh->t_full[b], 1);
            mbar_init(&sh->t_empty[b], SY_EW);
        }
        for (int b = 0; b < 2 * NC; ++b) mbar_init(&sh->c_full[b / NC][b % NC], 4);
        mbar_init(&sh->drain, 1);
        sh->abort = 0;
        fence_mbar_init();
    }
    __syncthreads();
    if (warp == 0) tmem_alloc(&sh->tbase, 512);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = sh->tbase;
    volatile int* abort = &sh->abort;
    auto give_up = [&]() {
        *abort = 1;
        atomicExch(err, 1);
    };
    const int run = blockIdx.x;
    int u = (int)sg.run_begin(run);
    const int u1 = (int)sg.run_begin(run + 1);
    int I = sg.block_of(u);

    if (warp == 0) {
        // ---------------------------------------------------------- producer
        if (lane == 0 && !stall_copies) {
            uint32_t ic = 0, cc = 0;
            bool ok = true;
            for (; u < u1 && ok && !*abort; ++I, ++ic) {
                const int uI = (int)sg.first(I), ue = min(u1, (int)sg.first(I + 1));
                const int nrt = sg.row_tiles(I);
                const int c0 = I * sg.RU + (u - uI), c1 = I * sg.RU + (ue - uI);
                auto column = [&](int c) {
                    const uint32_t s = cc & 1u;
                    if (!mbar_wait(&sh->b_empty[s], ((cc >> 1) & 1u) ^ 1u, wlimit)) { ok = false; return; }
                    mbar_expect_tx(&sh->b_full[s], CT * tileF + BN * 4u);
                    // CT feature tiles (BN > 128 only at one K slab, where they stack to BN rows)
                    bulk_g2s(sB + s * (CT * tileF), FB + (size_t)c * (CT * tileF), CT * tileF, &sh->b_full[s]);
                    bulk_g2s(sV + s * BN, Vp + (size_t)c * BN, BN * 4u, &sh->b_full[s]);
                    ++cc;
                };
                column(c0);
                for (int r = 0; r < nrt && ok; ++r) {
                    if (!mbar_wait(&sh->a_empty[r], (ic & 1u) ^ 1u, wlimit)) { ok = false; break; }
                    mbar_expect_tx(&sh->a_full[r], tileF);
                    bulk_g2s(sA + (size_t)r * tileF, FA + ((size_t)I * (R / SY_T) + r) * tileF, tileF,
                             &sh->a_full[r]);
                }
                for (int c = c0 + 1; c < c1 && ok; ++c) column(c);
                u = ue;
            }
            if (!ok) give_up();
            // every copy issued lands before the CTA may exit (each barrier's newest phase)
            for (uint32_t i = 0; i < min(cc, 2u); ++i)
                mbar_wait(&sh->b_full[(cc - 1 - i) & 1u], ((cc - 1 - i) >> 1) & 1u, wlimit);
            if (!ok || *abort) {
                // row tiles whose MMA may never have run; a phase that is past reports at once
                for (int r = 0; r < R / SY_T; ++r) {
                    if (ic > 0) mbar_wait(&sh->a_full[r], (ic - 1) & 1u, min(wlimit, 1LL << 24));
                    mbar_wait(&sh->a_full[r], ic & 1u, min(wlimit, 1LL << 24));
                }
            }
        }
    } else if (warp == 1) {
        // ---------------------------------------------------------- MMA issuer
        if (lane == 0) {
            const uint32_t idesc = idesc_bf16(SY_T, BN);
            // descriptors differ in the start address field alone (16-byte units): the issue loop
            // only adds to it.  Computing them in place cost ~175 cycles per MMA, next to four
            // epilogue warps on the same scheduler.
            const uint64_t ad0 = smem_desc_sw128(smem_u32(sA)), bd0 = smem_desc_sw128(smem_u32(sB));
            const uint32_t step = tileF >> 4;
            uint32_t koff[NK];                         // 64-wide slabs of 16 KB, 32 bytes per K step
#pragma unroll
            for (int kk = 0; kk < NK; ++kk) {
                const uint32_t ks = (korder >> (4 * kk)) & 15u;
                koff[kk] = (ks >> 2) * 1024u + (ks & 3u) * 2u;
            }
            uint32_t ic = 0, cc = 0, g = 0;
            bool ok = true, issued = false;
            for (; u < u1 && ok && !*abort; ++I, ++ic) {
                const int ue = min(u1, (int)sg.first(I + 1));
                const int nrt = sg.row_tiles(I);
                const int ncol = ue - u;
                for (int c = 0; c < ncol && ok; ++c, ++cc) {
                    const uint32_t s = cc & 1u;
                    if (!mbar_wait(&sh->b_full[s], (cc >> 1) & 1u, wlimit)) { ok = false; break; }
                    const uint64_t bd = bd0 + s * (CT * step);
                    for (int r = 0; r < nrt; ++r, ++g) {
                        const uint32_t b = g % NBUF;
                        if (c == 0 && !mbar_wait(&sh->a_full[r], ic & 1u, wlimit)) { ok = false; break; }
                        if (!mbar_wait(&sh->t_empty[b], ((g / NBUF) & 1u) ^ 1u, wlimit)) { ok = false; break; }
                        issued = true;
                        tc_fence_after();
                        const uint64_t ad = ad0 + (uint32_t)r * step;
                        const uint32_t dt = tmem + b * BN;
#pragma unroll
                        for (int kk = 0; kk < NK; ++kk) {
                            mma_bf16(dt, ad + koff[kk], bd + koff[kk], idesc, kk > 0 ? 1u : 0u);
                        }
                        mma_commit(&sh->t_full[b]);
                        if (c == ncol - 1) mma_commit(&sh->a_empty[r]);
                    }
                    if (ok) mma_commit(&sh->b_empty[s]);
                }
                u = ue;
            }
            if (!ok) give_up();
            if (issued) {   // no MMA writes TMEM any more once this phase completes
                mma_commit(&sh->drain);
                mbar_wait(&sh->drain, 0, wlimit);
            }
        }
    } else {
        // ---------------------------------------------------------- epilogue
        const int quarter = warp & 3, half = (warp - 2) >> 2;
        const int lr = lane >> 2, lc = 2 * (lane & 3);   // this thread's first row and column of a chunk
        const int lrow = quarter * 32 + lr + 8 * (lane & 3);   // the row whose sum it folds
        const uint32_t tb0 = tmem + ((uint32_t)(quarter * 32) << 16) + (uint32_t)(half * CW);
        uint32_t cc = 0, g = 0;
        bool dead = false;
        auto wait = [&](uint64_t* bar, uint32_t parity) {
            if (__all_sync(0xffffffffu, mbar_try_wait(bar, parity))) return;
            if (!dead) {
                bool ok = !*abort && mbar_wait(bar, parity, wlimit);
                ok = __all_sync(0xffffffffu, ok);
                if (!ok) {
                    dead = true;
                    if (lane == 0) give_up();
                }
            }
        };
        // column unit uc's sums over the four quarters; one warp of the half stores them
        auto store_column = [&](uint32_t uc, float2* out) {
            if (quarter != (int)(uc & 3u)) return;
            wait(&sh->c_full[half][uc % NC], (uc / NC) & 1u);
            const float* col = sCol + (uc % NC) * (4 * BN) + half * CW + lane;
#pragma unroll
            for (int j = 0; j < NQ; ++j) {
                float2 x = make_float2(0.f, 0.f);
#pragma unroll
                for (int w = 0; w < 4; ++w) ff_add(x.x, x.y, col[w * BN + 32 * j]);
                out[half * CW + 32 * j + lane] = x;
            }
        };
        // v is scaled by the power of two that puts max |v| in [2^14, 2^15) (products and sums of
        // tiny or huge v stay in range); vscale undoes it in the reduction
        float vs2;
        {
            float m = 0.f;
            for (int j = lane; j < nbmax; j += 32) m = fmaxf(m, bmax[j]);
            m = warp_max(m);
            int ex = 15;
            if (m > 0.f && m <= 3.4028234663852886e38f) frexpf(m, &ex);
            const int ev = max(-126, min(126, 15 - ex));
            vs2 = ldexpf(1.f, ev);
            if (run == 0 && warp == 2 && lane == 0) *vscale = ldexp(1.0, -ev);
        }
        uint32_t nc = 0;                           // column units that gave column sums
        float2* prev = nullptr;
        // Chunks of 16 rows x 32 columns run through four register sets in three stages: one is
        // being loaded, the next exponentiated (in place), the one before multiplied.  Stages of
        // one step are independent, so that the MUFU and FMA streams interleave.
        constexpr int NCH = 2 * NQ;                // chunks per tile: column chunk i / 2, row half i % 2
        uint32_t t[4][16];
        auto load = [&](uint32_t b, int i, uint32_t (&x)[16]) {
            tmem_ld_16x32(tb0 + ((uint32_t)(16 * (i & 1)) << 16) + b * BN + 32u * (i >> 1), x);
        };
        auto expo = [&](uint32_t (&x)[16]) {
#pragma unroll
            for (int k = 0; k < 16; ++k) x[k] = __float_as_uint(ex2f(__uint_as_float(x[k])));
        };
        wait(&sh->t_full[0], 0);                   // every run has a pair
        tc_fence_after();
        load(0, 0, t[0]);
        tmem_wait_ld16(t[0]);
        load(0, 1, t[1]);
        expo(t[0]);
        // Carried over to the next tile, whose exponentials hide their shuffles and adds: the row
        // sums of the last tile (pend, for the running sum at pend_at) and, at the start of a
        // unit, the column sums of the unit before (acc; slot_at is null when they are not used).
        float pend[4] = {0.f, 0.f, 0.f, 0.f};
        float2* pend_at = sRow + half * R + lrow;
        bool pend_first = true;
        unsigned long long acc[4 * NQ], v2[4 * NQ];
        float2* slot_at = nullptr;
#pragma unroll
        for (int k = 0; k < 4 * NQ; ++k) acc[k] = 0ull;
        // column chunk q's sums over the eight row groups: this thread ends with one of the 32
        // columns, the one that its lane bits select
        auto column_sum = [&](int q) {
            float a[8];
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                sy_unpack(acc[4 * q + k], a[2 * k], a[2 * k + 1]);
                acc[4 * q + k] = 0ull;
            }
            lane_sum<8, 16>(a, lane);
            sCol[(nc % NC) * (4 * BN) + quarter * BN + half * CW + 32 * q + 8 * (lane >> 3) + lc +
                 ((lane >> 2) & 1)] = a[0];
        };
        // Hands the unit's sums on.  The unit before that is complete by now or nearly so, and is
        // stored.  A buffer is written again NC units later: at most NBUF tiles lie between
        // two warps, and a unit has RT >= 2 of them, so that by then every warp has released a
        // tile past the one in which it read the buffer ((NC - 1) RT - 1 >= NBUF).
        auto column_done = [&]() {
            if (!slot_at) return;
            __syncwarp();
            if (lane == 0) mbar_arrive(&sh->c_full[half][nc % NC]);
            if (nc > 0) store_column(nc - 1, prev);
            prev = slot_at;
            ++nc;
        };
        for (; u < u1; ++I) {
            const int uI = (int)sg.first(I), ue = min(u1, (int)sg.first(I + 1));
            const int nrt = sg.row_tiles(I);
            const int ct0 = I * sg.RU + (u - uI), ncol = ue - u;
            const float* vrow = Vp + (size_t)I * R + quarter * 32 + lr;
            float2* srow = sRow + half * R + lrow;
            float2* cout = colpart + sg.col_base(ct0) + (long long)sg.slot(I) * BN;   // this unit's slot
            int cb = ct0 / sg.RU, cr = ct0 % sg.RU;
            float vn[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) vn[j] = __ldg(vrow + 8 * j);
            for (int c = 0; c < ncol; ++c, ++cc) {
                const uint32_t s = cc & 1u;
                const float* vs = sV + s * BN + half * CW + lc;
                wait(&sh->b_full[s], (cc >> 1) & 1u);
                auto tile = [&](int r, auto first) {
                    constexpr bool FIRST = decltype(first)::value;   // the unit's first tile
                    const uint32_t b = g % NBUF, bn = (g + 1) % NBUF;
                    const bool more = r + 1 < nrt || c + 1 < ncol || ue < u1;
                    float vr[4];                   // this tile's v; the next one's on its way
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        vr[j] = vn[j] * vs2;
                        vn[j] = __ldg(vrow + (r + 1 < nrt ? r + 1 : 0) * SY_T + 8 * j);
                    }
                    bool ready = true;
                    float2 h = pend_first ? make_float2(0.f, 0.f) : *pend_at;
                    unsigned long long rs[4] = {0ull, 0ull, 0ull, 0ull};
#pragma unroll
                    for (int i = 0; i < NCH; ++i) {
                        const int q = i / 2, hf = i % 2;
                        tmem_wait_ld16(t[(i + 1) & 3]);
                        // whether the next tile is there: asked a step ahead, off the critical path
                        if (i == NCH - 3) ready = !more || mbar_test_wait(&sh->t_full[bn], ((g + 1) / NBUF) & 1u);
                        if (i == NCH - 2) {
                            // this tile's last chunk has landed
                            tc_fence_before();
                            __syncwarp();
                            if (lane == 0) mbar_arrive(&sh->t_empty[b]);
                            // after the run's last tile this reads a buffer nobody fills any
                            // more, and the values are not used
                            if (more && !__all_sync(0xffffffffu, ready))
                                wait(&sh->t_full[bn], ((g + 1) / NBUF) & 1u);
                            tc_fence_after();
                        }
                        if (i < NCH - 2) load(b, i + 2, t[(i + 2) & 3]);
                        else load(bn, i + 2 - NCH, t[(i + 2) & 3]);
                        expo(t[(i + 1) & 3]);
                        if (FIRST && hf == 0) {
                            column_sum(q);
#pragma unroll
                            for (int k = 0; k < 4; ++k) {
                                const float2 v = *reinterpret_cast<const float2*>(vs + 32 * q + 8 * k);
                                v2[4 * q + k] = sy_pack(v.x * vs2, v.y * vs2);
                            }
                        }
                        const unsigned long long va = sy_pack(vr[2 * hf], vr[2 * hf]);
                        const unsigned long long vb = sy_pack(vr[2 * hf + 1], vr[2 * hf + 1]);
                        const uint32_t* x = t[i & 3];
#pragma unroll
                        for (int k = 0; k < 4; ++k) {
                            const unsigned long long pa = sy_pack(__uint_as_float(x[4 * k]), __uint_as_float(x[4 * k + 1]));
                            const unsigned long long pb =
                                sy_pack(__uint_as_float(x[4 * k + 2]), __uint_as_float(x[4 * k + 3]));
                            sy_fma(acc[4 * q + k], pa, va);
                            sy_fma(rs[2 * hf], pa, v2[4 * q + k]);
                            sy_fma(acc[4 * q + k], pb, vb);
                            sy_fma(rs[2 * hf + 1], pb, v2[4 * q + k]);
                        }
                        if (i == 1) {
                            // the last tile's rows lr + 8 j over the four threads that share
                            // them; this thread ends with j = lane % 4 and folds that row
                            lane_sum<4, 2>(pend, lane);
                            ff_add(h.x, h.y, pend[0]);
                            *pend_at = h;
                        }
                    }
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        float lo, hi;
                        sy_unpack(rs[j], lo, hi);
                        pend[j] = lo + hi;
                    }
                    pend_at = srow + r * SY_T;
                    pend_first = c == 0;
                    ++g;
                };
                tile(0, std::true_type{});
                __syncwarp();
                if (lane == 0) mbar_arrive(&sh->b_empty[s]);
                column_done();
                slot_at = cb > I ? cout : nullptr;   // right of the diagonal block
                cout += (long long)sg.slots(cb) * BN;
                if (++cr == sg.RU) {
                    cr = 0;
                    ++cb;
                }
#pragma unroll 1
                for (int r = 1; r < nrt; ++r) tile(r, std::false_type{});
            }
            // the piece's last row sums, then both column halves of every row
            float2 h = pend_first ? make_float2(0.f, 0.f) : *pend_at;
            lane_sum<4, 2>(pend, lane);
            ff_add(h.x, h.y, pend[0]);
            *pend_at = h;
            sy_bar(1, 32 * SY_EW);
            for (int row = tid - 64; row < nrt * SY_T; row += 32 * SY_EW) {
                float2 x = sRow[row];
                const float2 y = sRow[R + row];
                ff_add(x.x, x.y, y.x);
                x.y += y.y;
                rowpart[(long long)(run + sg.slot(I)) * R + row] = x;
            }
            sy_bar(1, 32 * SY_EW);
            // nothing is pending: the next fold writes a zero where the next piece starts anew
#pragma unroll
            for (int j = 0; j < 4; ++j) pend[j] = 0.f;
            pend_at = srow;
            pend_first = true;
            u = ue;
        }
#pragma unroll
        for (int q = 0; q < NQ; ++q) column_sum(q);
        column_done();
        if (nc > 0) store_column(nc - 1, prev);
        tmem_wait_ld16(t[1]);
    }
    __syncwarp();
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (warp == 0) tmem_dealloc(tmem, 512);
}

// q_i = ksc vscale (sum of point i's column and row slots) + beta v_i (vscale null: 1).  One block per tile: 128 points
// x 4 interleaved groups of column slots.  With cg also v . q, in whose last block the CG step is formed:
// a pass of its own over both vectors cost an iteration 5 us (58 of them at n = 6000, k = 200).
// A float pair that overflowed, or met an infinity, holds Inf - Inf in its low half, and a sum of both
// signs may overflow on the way to a finite value.  Points with such a slot are summed again from the
// points themselves in FP64, where the kernel has them (pts.P: FP32 products; the tensor-core product
// scales v, so that only an infinity in v gets there, and takes the high half): exact-form
// semantics for the price of one flag a block otherwise.
constexpr int SYR_G = 4;
__device__ __noinline__ double sy_exact_sum(SyPoints pts, const float* V, int n, int i, int j0) {
    double s = 0.0;
    const float* x = pts.P + (size_t)i * pts.ps;
    for (int j = j0; j < n; j += SYR_G) {
        const float* y = pts.P + (size_t)j * pts.ps;
        float t = pts.nsc != 0.f ? 0.f : x[pts.d] + y[pts.d];
        for (int c = 0; c < pts.d; ++c)
            t = pts.nsc != 0.f ? fmaf(x[c] - y[c], x[c] - y[c], t) : fmaf(2.f * x[c], y[c], t);
        s = fma((double)ex2f(pts.nsc != 0.f ? pts.nsc * t : t), (double)V[j], s);
    }
    return s;
}
// With panels acc holds the sums of those before (the first writes it), and Q is written after the last.
template <class Grid>
__global__ void __launch_bounds__(SY_T * SYR_G)
k_sym_reduce(Grid sg, const float2* __restrict__ rowpart, const float2* __restrict__ colpart,
             const float* __restrict__ V, float beta, double ksc, const double* __restrict__ vscale,
             float* __restrict__ Q, CGScalars* cg, double* __restrict__ dpart, SyPoints pts, double* __restrict__ acc) {
    pdl_entry();
    __shared__ double red[SYR_G][SY_T];
    __shared__ double dred[SY_T / 32];
    const int x = threadIdx.x & (SY_T - 1), grp = threadIdx.x / SY_T;
    const int i = blockIdx.x * SY_T + x;
    const int T = i / sg.BN, b = T / sg.RU;
    const float2* cp = colpart + sg.col_base(T) + i % sg.BN;
    const int nslot = sg.slots(b);
    float h = 0.f, l = 0.f;
#pragma unroll 4
    for (int I = grp; I < nslot; I += SYR_G) {
        const float2 w = cp[(long long)I * sg.BN];
        ff_add(h, l, w.x);
        l += w.y;
    }
    if (sg.has(b)) {
        const int s0 = sg.run_of(sg.first(b)), s1 = sg.run_of(sg.first(b + 1) - 1);
        for (int s = s0 + grp; s <= s1; s += SYR_G) {
            const float2 w = rowpart[(long long)(s + sg.slot(b)) * sg.rows() + i % sg.rows()];
            ff_add(h, l, w.x);
            l += w.y;
        }
    }
    bool over = !(fabsf(h) <= 3.402823466e38f);
    double v64 = over ? (double)h : (double)h + (double)l;
    if (!sg.first_panel() && grp == 0 && i < sg.n) {
        v64 += acc[i];
        over = over || !isfinite(v64);             // a panel before was
    }
    red[grp][x] = v64;
    const bool last = sg.last_panel();
    if (__syncthreads_or(over && last && pts.P)) {   // rare
        double t = 0.0;
#pragma unroll
        for (int w = 0; w < SYR_G; ++w) t += red[w][x];
        const bool redo = i < sg.n && !isfinite(t);
        __syncthreads();
        if (redo) red[grp][x] = sy_exact_sum(pts, V, sg.n, i, grp);
        __syncthreads();
    }
    double dot = 0.0;
    if (grp == 0 && i < sg.n) {
        double t = red[0][x];
#pragma unroll
        for (int w = 1; w < SYR_G; ++w) t += red[w][x];
        if (!last) {
            acc[i] = t;
            return;
        }
        const float v = V[i];
        const float q = (float)(t * (vscale ? ksc * *vscale : ksc) + (beta != 0.f ? (double)beta * v : 0.0));
        Q[i] = q;
        dot = (double)v * (double)q;
    }
    if (!cg || !last) return;
    if (grp == 0) {
        dot = warp_sum(dot);
        if ((x & 31) == 0) dred[x >> 5] = dot;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        double t = 0.0;
#pragma unroll
        for (int w = 0; w < SY_T / 32; ++w) t += dred[w];
        dpart[blockIdx.x] = t;
    }
    if (!last_block(&cg->ticket[1]) || threadIdx.x >= 32) return;
    const double t = warp_sum_parts(dpart, gridDim.x, 0);
    if (threadIdx.x == 0) cg_alpha(cg, 0, t);
}

template <class Grid>
int launch_sym_reduce(krr_ctx* ctx, const Grid& g, const float2* rowpart, const float2* colpart, const float* V,
                      float beta, double ksc, const double* vscale, float* Q, SyPoints pts) {
    const int blocks = g.NU * g.BN / SY_T;
    const bool pq = ctx->want_pq && g.last_panel();
    double *dpart = nullptr, *acc = nullptr;
    if (pq) KRR_RET(bufT(ctx, "sym_dot", (size_t)blocks, &dpart));
    if (!g.first_panel() || !g.last_panel()) KRR_RET(bufT(ctx, "sym_acc", (size_t)g.n, &acc));
    launch_pdl(&k_sym_reduce<Grid>, blocks, SY_T * SYR_G, 0, ctx->stream, g, rowpart, colpart, V, beta, ksc, vscale, Q,
               dpart ? ctx->cg : nullptr, dpart, pts, acc);
    KRR_CHECK_LAUNCH();
    ctx->have_pq = pq;
    return KRR_OK;
}
template int launch_sym_reduce(krr_ctx*, const SyGrid&, const float2*, const float2*, const float*, float, double,
                               const double*, float*, SyPoints);
template int launch_sym_reduce(krr_ctx*, const SyPanel&, const float2*, const float2*, const float*, float, double,
                               const double*, float*, SyPoints);

int sym_buffers(krr_ctx* ctx, const SyGrid& g, void** row, void** col) {
    const size_t nr = 8 * (size_t)(g.G + g.nblk) * g.rows();
    const size_t nc = 8 * (size_t)std::min<long long>(g.col_base(g.NU), kSymBytes / 8);
    if (ctx->sym_nomem && nr + nc >= ctx->sym_nomem)
        return fail(ctx, KRR_E_NOMEM, "symmetric product: no room for its partial sums");
    int rc = buf(ctx, "sy_row", nr, row);
    if (rc == KRR_OK) rc = buf(ctx, "sy_col", nc, col);
    if (rc == KRR_E_NOMEM) ctx->sym_nomem = nr + nc;
    return rc;
}

static size_t sym_smem(int Kp, int BN, int RU) {
    const size_t tileF = 128u * (size_t)Kp * 2u;
    const size_t rt = (size_t)RU * BN / SY_T;
    return 1024 + (rt + 2 * BN / SY_T) * tileF + 2 * (size_t)BN * 4 + 2 * rt * SY_T * 8 +
           (size_t)sy_nc(BN) * 4 * BN * 4 + sizeof(SyShared);
}

double ex2_bias_scale(const krr_ctx* ctx);

// K steps in the order they are issued, a nibble each: those with the fewest leading products (2 x_i x_j of
// a coordinate, at feature 6 c) first, the norms (feature 6 d + 3 is the leading piece of the later one)
// last.  A step rounds downwards at the size of the partial sum, and the sum climbs to 2 x_i . x_j before
// the norms are taken off, so it should climb late.  Relative error on clusters far from the centre (the
// mixture, n = 3000) in the features' order and in this one, beside the 5.60e-6 and 14.5e-6 of the product
// of two sets, which carries v in the exponent: d = 8 5.67e-6 and 5.04e-6, d = 12 14.5e-6 and 13.3e-6;
// within 2% either way for points about the centre, at a tenth of that product's error.  The norms in the
// middle: 2.0e-6 at d = 8, but 1.3e-7 instead of 0.95e-7 for N(0, I), where solves near the limit of the
// precision (n = 30000, beta = 1e-3) then took half as many iterations again.
static uint32_t sym_korder(int dk, int nk) {
    const int norms = (6 * dk + 3) / 16;
    int key[8];
    for (int k = 0; k < nk; ++k) {
        key[k] = k >= norms ? 16 + k : 0;
        for (int c = 0; c < dk && k < norms; ++c) key[k] += 6 * c / 16 == k;
    }
    uint32_t o = 0, taken = 0;
    for (int i = 0; i < nk; ++i) {
        int best = -1;
        for (int k = 0; k < nk; ++k)
            if (!((taken >> k) & 1u) && (best < 0 || key[k] < key[best])) best = k;
        taken |= 1u << best;
        o |= (uint32_t)best << (4 * i);
    }
    return o;
}

template <class Grid>
using sym_fn = void (*)(const unsigned char*, const unsigned char*, int, Grid, const float*, float2*, float2*,
                        const float*, int, double*, int*, long long, int, uint32_t);
template <class Grid>
static sym_fn<Grid> sym_pick(int nk) {
    switch (nk) {
        case 1: return &k_kmvm_sym<1, 256, Grid>;
        case 2: return &k_kmvm_sym<2, 256, Grid>;
        case 3: return &k_kmvm_sym<3, 256, Grid>;
        case 4: return &k_kmvm_sym<4, 256, Grid>;
        case 5: return &k_kmvm_sym<5, 128, Grid>;
        case 6: return &k_kmvm_sym<6, 128, Grid>;
        case 7: return &k_kmvm_sym<7, 128, Grid>;
    }
    return nullptr;
}

// Whether the symmetric form takes a square product of n points: it is the faster one at every
// size measured; past the limit k_kmvm_tc runs.
bool sym_tc_fits(long long n) { return n <= (1LL << 21); }

int launch_kmvm_sym(krr_ctx* ctx, const unsigned char* FA, const unsigned char* FB, long long n, int d,
                    float beta, const float* V, float* Q, int* err) {
    const int Kp = tc_feature_kp(d);
    const int nk = (6 * kernel_dim(d) + 6 + 15) / 16;   // K steps that hold features
    // 128-wide features (d >= 10) leave room for two 128-column stages only
    const int BN = Kp == 64 ? 256 : 128;
    const int rumin = 2 * SY_T / BN, rumax = (Kp == 64 ? SY_RTMAX : 4) * SY_T / BN;   // by shared memory
    if (!sym_pick<SyGrid>(nk)) return fail(ctx, KRR_E_INVAL, "symmetric product: unsupported dimension");
    auto make = [&](int RU) {
        SyGrid g{};
        g.n = (int)n;
        g.BN = BN;
        g.NU = (int)ceil_div(n, BN);
        g.RU = RU;
        g.nblk = (g.NU + RU - 1) / RU;
        g.W = g.first(g.nblk);
        g.G = (int)std::min<long long>(g.W, ctx->num_sms);
        return g;
    };
    // units per row block: the longest run sets the time, so minimise pairs per run x (row tiles
    // per pair + the pair's lane reduction, about half a tile)
    int best = rumin;
    double best_cost = 0.0;
    for (int RU = rumin; RU <= rumax; ++RU) {
        const SyGrid g = make(RU);
        const double cost = (double)((g.W + g.G - 1) / g.G) * (RU * BN / SY_T + 0.5);
        if (RU == rumin || cost < best_cost) {
            best_cost = cost;
            best = RU;
        }
    }
    const int RU = std::max(rumin, tuned_splits(ctx, tune_key(kFormSym, Kp, 1, n), best, rumax));
    ctx->last_splits = RU;
    const SyGrid g = make(RU);
    const int np = g.NU * BN;
    const int nbmax = (int)ceil_div(np, SY_PAD);
    float *Vp, *bmax;
    double* vscale;
    KRR_RET(bufT(ctx, "sy_vp", (size_t)np, &Vp));
    KRR_RET(bufT(ctx, "sy_bmax", (size_t)nbmax, &bmax));
    KRR_RET(bufT(ctx, "sy_vsc", 1, &vscale));
    const long long wlimit = ctx->opts.wait_limit_log2 > 0 ? (1LL << ctx->opts.wait_limit_log2)
                                                           : kWaitLimitDefault;
    const size_t smem = std::max<size_t>(sym_smem(Kp, BN, RU), 120 * 1024);   // one CTA per SM (TMEM)
    const uint32_t korder = sym_korder(kernel_dim(d), nk);
    bool padded = false;
    return sym_product(ctx, g, [&](const auto& p, void* row, void* col) -> int {
        using Grid = std::decay_t<decltype(p)>;
        const sym_fn<Grid> fn = sym_pick<Grid>(nk);
        float2 *rowpart = (float2*)row, *colpart = (float2*)col;
        KRR_RET(allow_max_dynamic_smem(ctx, (const void*)fn));
        if (!padded) {
            launch_pdl(k_sym_pad, nbmax, SY_PAD, 0, ctx->stream, V, (int)n, np, Vp, bmax);
            KRR_CHECK_LAUNCH();
            padded = true;
        }
        launch_pdl(fn, p.G, SY_THREADS, smem, ctx->stream, FA, FB, Kp, p, Vp, rowpart, colpart, bmax, nbmax, vscale, err,
                   wlimit, ctx->opts.test_stall_copies, korder);
        KRR_CHECK_LAUNCH();
        return launch_sym_reduce(ctx, p, rowpart, colpart, V, beta, ex2_bias_scale(ctx), vscale, Q, SyPoints());
    });
}

}  // namespace krr

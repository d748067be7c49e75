// Tensor-core K.V on symmetric tile pairs, FP32 (the inner product of the
// mixed-precision solver, KPCG_TC_IR, for one column at a time).
//
// The entries are those of kv_tc_kernel: the BF16x3 augmented operands of
// tc_prep_kernel give the exp2 argument a_ij = log2(s^2) - |x'_i - x'_j|^2 of
// Eq. 1 in an FP32 accumulator, exp2 runs on the MUFU.  K is symmetric, so
// each pair of 128-point tiles (I, c), I <= c, is evaluated once: it
// gives the row sums K_Ic V_c for the rows of I and, from the same entries,
// the column sums K_Ic^T V_I for the rows of c (not for I = c, whose tile is
// evaluated in full and gives row sums only).
//
// A column tile J of 256 points (c = 2 J and 2 J + 1) is the CTA's resident operand
// (B in shared memory for the whole work item) and the row tiles I stream through a
// ring (A tile and V_I per stage).  Each epilogue thread owns one row of the
// tile and 64 of its columns: per entry one TMEM word, one ex2, one FMA into
// its row sum (V_j by broadcast from shared memory, four at a time) and one FMA into
// its column accumulator in registers (V_i, one value per tile) -- no shuffles per
// entry.  The column accumulators are reduced over the 128 rows once per work
// item (a shuffle butterfly, then the four row quarters through shared
// memory); the four column groups' row sums are added through shared memory by a
// warp of their own.  Row sums leave once per (I, J), column sums once per
// work item; a second kernel adds, for every point, its row partials and the
// column partials of its tile in a fixed order.
//
// Roles (20 warps, one CTA per SM): warps 0..15 are the epilogue (row quarter =
// warp mod 4, the TMEM lanes a warp may read; column group = warp / 4), warp 16
// bulk-copies (the B tile once, then A tiles and V_I into a 4-stage ring), warp 17
// issues the MMAs from one thread into double-buffered TMEM accumulators, warp
// 18 adds the row sums, warp 19 only keeps the count a multiple of four.  A tile costs
// an epilogue warp one wait and one arrival: the arrival says that the accumulator,
// the stage and the row-sum slot of the tile are done with.  Every wait is bounded.
//
// What bounds it: the MUFU (32 ex2 per clock and SM) is 44% busy and issue 63% (ncu,
// n = 65536); the rest is latency of the ex2 and TMEM reads.  Eight warps on tiles of 128
// columns with V_J in registers took 514 us for this kernel against 517 here, but write
// four times the row partials; sixteen warps of 32 columns 571 us.  With the reduction
// below n = 65536, d = 8 takes 0.57 ms per product (0.82 ms with an FP64 reduction, a
// load and a wait per 16 columns and the MMAs issued by one lane).
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <vector>

#include "ctx.cuh"
#include "tcgen05.cuh"

namespace kpcg {
namespace {

constexpr int SN = 2 * TN;                // columns per column tile (MMA N)
constexpr int SEPI_TCS = 16;              // epilogue warps
constexpr int SWARPS_TCS = SEPI_TCS + 4;  // + producer, MMA issuer, row sums, none
constexpr int SCOLS = 64;                 // columns per epilogue thread
constexpr int SGRP = SN / SCOLS;          // column groups
constexpr int STAGES_TCS = 4;

template <int KCH>
struct TcsSmem {
    static constexpr uint32_t kSub = SUB * 2;                           // 16 KB
    static constexpr uint32_t kB = KCH * 2 * kSub;                      // resident B tile
    static constexpr uint32_t kAst = KCH * kSub;                        // A part of a stage
    static constexpr uint32_t kStage = ((kAst + TM * 4 + 1023) / 1024) * 1024;  // + V_I
    static constexpr uint32_t kV = SN * 4;                              // V_J
    static constexpr uint32_t kCol = 4 * SN * 4;                        // [quarter][column]
    static constexpr uint32_t kRow = STAGES_TCS * SGRP * TM * 4;        // [slot][group][row]
    static constexpr uint32_t kBars = 1024;
    static constexpr uint32_t kTotal = 1024 + kB + STAGES_TCS * kStage + kV + kCol + kRow + kBars;
};

// kind::f16 instruction descriptor: BF16 x BF16 -> FP32, K-major, M = 128, N = SN.
constexpr uint32_t kIdescN = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(SN >> 3) << 17) |
                             ((uint32_t)(TM >> 4) << 24);

// Sums 64 values per lane (columns 0..63, one row per lane) over the 32
// lanes: five halving steps across lane bits 16, 8, 4, 2, 1, each sending
// half of the columns a lane holds to its partner and adding the other half
// to the partner's copy, leave in lane l the sums over all 32 rows of columns 2 l
// and 2 l + 1 in v[0] and v[1].
__device__ __forceinline__ void tcs_colsum64(float (&v)[64], int lane) {
#pragma unroll
    for (int w = 64, m = 16; w > 2; w >>= 1, m >>= 1) {
        const bool u = (lane & m) != 0;
        const int hw = w >> 1;
#pragma unroll
        for (int q = 0; q < hw; ++q) {
            const float snd = u ? v[q] : v[q + hw];
            const float kep = u ? v[q + hw] : v[q];
            v[q] = kep + __shfl_xor_sync(0xffffffffu, snd, m);
        }
    }
}

// Index of the row partials of row tile I and column tile J (256 columns: the tiles
// 2 J and 2 J + 1 of 128), I <= 2 J + 1.
__host__ __device__ __forceinline__ int64_t tcs_pair(int64_t J, int64_t I) {
    return J * (J + 1) + I;
}

template <int KCH>
__global__ void __launch_bounds__(SWARPS_TCS * 32, 1)
    kv_tcs_kernel(const __nv_bfloat16* __restrict__ Aop, const __nv_bfloat16* __restrict__ Bop,
                  const float* __restrict__ Vs, int64_t n_t, const int4* __restrict__ work,
                  float* __restrict__ prow, float* __restrict__ pcol, int* __restrict__ err,
                  uint64_t wait_ns, int stall) {
    using S = TcsSmem<KCH>;
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = reinterpret_cast<uint8_t*>(
        (reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    uint8_t* sB = smem;
    uint8_t* sStage = smem + S::kB;
    float* sV = reinterpret_cast<float*>(sStage + STAGES_TCS * S::kStage);
    float* colbuf = sV + SN;
    float* rowbuf = colbuf + 4 * SN;
    uint64_t* bars = reinterpret_cast<uint64_t*>(rowbuf + STAGES_TCS * SGRP * TM);
    uint64_t* full = bars;                   // [STAGES] copies landed
    uint64_t* used = full + STAGES_TCS;      // [STAGES] the epilogue is done with a tile
    uint64_t* summed = used + STAGES_TCS;    // [STAGES] its row sums are added
    uint64_t* tfull = summed + STAGES_TCS;   // [2] accumulator ready
    uint64_t* bfull = tfull + 2;
    uint64_t* done = bfull + 1;
    uint64_t* never = done + 1;  // test hook: no thread ever arrives here
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(never + 1);
    __shared__ int s_fail;

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int4 wk = work[blockIdx.x];
    const int64_t J = wk.x;
    const int64_t I0 = wk.y;
    const int ntiles = wk.z - wk.y;
    const bool two = 2 * J + 1 < n_t;  // the second 128 columns exist

    if (threadIdx.x < SN)
        sV[threadIdx.x] = (threadIdx.x < TN || two) ? Vs[(size_t)J * SN + threadIdx.x] : 0.f;
    if (threadIdx.x == 0) {
        for (int s = 0; s < STAGES_TCS; ++s) {
            mbar_init(&full[s], 1);
            mbar_init(&used[s], SEPI_TCS);
            mbar_init(&summed[s], 1);
        }
        mbar_init(&tfull[0], 1);
        mbar_init(&tfull[1], 1);
        mbar_init(bfull, 1);
        mbar_init(done, 1);
        mbar_init(never, 1);
        s_fail = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == SEPI_TCS + 1) {
        asm volatile(
            "tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                su32(tmem_slot)),
            "r"(2 * SN));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    fence_before();
    __syncthreads();
    fence_after();
    const uint32_t tmem = *tmem_slot;
    const uint64_t deadline = gtimer() + wait_ns;
    int fail = 0;

    if (warp == SEPI_TCS) {
        if (lane == 0) {
            mbar_expect_tx(bfull, (two ? 2 : 1) * KCH * S::kSub);
            for (int h = 0; h < (two ? 2 : 1); ++h)
                for (int kc = 0; kc < KCH; ++kc)  // 256 rows of each K sub-tile together
                    bulk_g2s(sB + (size_t)(kc * 2 + h) * S::kSub,
                             Bop + (size_t)((2 * J + h) * KCH + kc) * SUB, S::kSub, bfull);
            int t = 0;
            for (; t < ntiles; ++t) {
                const int s = t % STAGES_TCS;
                const uint32_t ph = ((uint32_t)(t / STAGES_TCS) & 1u) ^ 1u;
                if (!mbar_wait_idle(&used[s], ph, deadline) ||
                    !mbar_wait_idle(&summed[s], ph, deadline)) {
                    fail = 1;
                    break;
                }
                const int64_t it = I0 + t;
                uint8_t* st = sStage + (size_t)s * S::kStage;
                mbar_expect_tx(&full[s], S::kAst + TM * 4);
                bulk_g2s(st, Aop + (size_t)it * KCH * SUB, S::kAst, &full[s]);
                bulk_g2s(st + S::kAst, Vs + (size_t)it * TM, TM * 4, &full[s]);
            }
            // the CTA exits only once the copies it issued have landed
            const uint64_t dl2 = gtimer() + 200000000ull;
            for (int q = (t > STAGES_TCS ? t - STAGES_TCS : 0); q < t; ++q)
                (void)mbar_wait(&full[q % STAGES_TCS], (uint32_t)(q / STAGES_TCS) & 1u, dl2);
            (void)mbar_wait(bfull, 0, dl2);
        }
    } else if (warp == SEPI_TCS + 1) {
        const uint32_t el = elect_one();
        // test hook: a wait on a barrier nothing arrives at runs out
        if (stall && !mbar_wait_warp(never, 0, deadline)) fail = 1;
        if (!fail && !mbar_wait_warp(bfull, 0, deadline)) fail = 1;
        fence_after();
        const uint32_t b0 = su32(sB);
        const uint32_t idesc = two ? kIdescN : kIdesc;
        for (int t = 0; t < ntiles && !fail; ++t) {
            const int s = t % STAGES_TCS, b = t & 1, u = t - 2;
            if (!mbar_wait_warp(&full[s], (uint32_t)(t / STAGES_TCS) & 1u, deadline) ||
                (u >= 0 && !mbar_wait_warp(&used[u % STAGES_TCS],
                                           (uint32_t)(u / STAGES_TCS) & 1u, deadline))) {
                fail = 1;
                break;
            }
            fence_after();
            const uint32_t a0 = su32(sStage + (size_t)s * S::kStage);
            const uint32_t dt = tmem + (uint32_t)(b * SN);
#pragma unroll
            for (int kc = 0; kc < KCH; ++kc)
#pragma unroll
                for (int kk = 0; kk < KC / 16; ++kk)
                    mma_ss(dt, sdesc(a0 + (uint32_t)kc * S::kSub + (uint32_t)kk * 32),
                           sdesc(b0 + (uint32_t)kc * 2 * S::kSub + (uint32_t)kk * 32), idesc,
                           (kc | kk) ? 1u : 0u, el);
            mma_commit(&tfull[b], el);
        }
        mma_commit(done, el);
        if (!mbar_wait_warp(done, 0, gtimer() + kWaitNs)) fail = 1;
    } else if (warp == SEPI_TCS + 2) {
        // row sums of a tile: the column groups' in a fixed order
        float* out = prow + tcs_pair(J, I0) * TM;
        for (int t = 0; t < ntiles; ++t, out += TM) {
            const int s = t % STAGES_TCS;
            if (!__all_sync(0xffffffffu, mbar_wait_idle(&used[s], (uint32_t)(t / STAGES_TCS) & 1u, deadline))) {
                fail = 1;
                break;
            }
            const float* rb = rowbuf + s * SGRP * TM;
#pragma unroll
            for (int r = lane; r < TM; r += 32)
                out[r] = (rb[r] + rb[TM + r]) + (rb[2 * TM + r] + rb[3 * TM + r]);
            __syncwarp();
            if (lane == 0) mbar_arrive(&summed[s]);
        }
    } else if (warp < SEPI_TCS) {
        const int quarter = warp & 3;
        const int grp = warp >> 2;                 // columns 64 grp .. + 63
        const int row = quarter * 32 + lane;
        const int64_t ct = 2 * J + (grp >> 1);     // their tile of 128
        float cs[SCOLS];  // column sums over the row tiles of the item
#pragma unroll
        for (int j = 0; j < SCOLS; ++j) cs[j] = 0.f;
        const uint32_t vj = su32(sV + grp * SCOLS);
        const uint32_t tbase =
            tmem + ((uint32_t)(quarter * 32) << 16) + (uint32_t)(grp * SCOLS);
        for (int t = 0; t < ntiles; ++t) {
            const int s = t % STAGES_TCS, b = t & 1;
            if (!mbar_wait_warp(&tfull[b], (uint32_t)(t >> 1) & 1u, deadline)) {
                fail = 1;
                break;
            }
            fence_after();
            const int64_t it = I0 + t;
            float sum = 0.f;
            if (it <= ct && ct < n_t) {  // (a row tile below its column tile is the other's)
                // chunks of 8 columns, the next one's load in flight while a chunk is
                // evaluated
                uint32_t r0[8], r1[8];
                auto ld = [&](int ps, uint32_t (&r)[8]) {
                    asm volatile(
                        "tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, "
                        "[%8];"
                        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]),
                          "=r"(r[6]), "=r"(r[7])
                        : "r"(tbase + (uint32_t)(b * SN + ps * 8)));
                };
                auto arrived = [&](uint32_t (&r)[8]) {
                    asm volatile("tcgen05.wait::ld.sync.aligned;"
                                 : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]),
                                   "+r"(r[5]), "+r"(r[6]), "+r"(r[7])
                                 :
                                 : "memory");
                };
                ld(0, r0);
                // the diagonal tile gives row sums only: its column sums get zeros
                const float vi =
                    it < ct ? lds32(su32(sStage + (size_t)s * S::kStage + S::kAst) + row * 4) : 0.f;
                float a[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
                for (int ps = 0; ps < SCOLS / 8; ++ps) {
                    uint32_t (&r)[8] = (ps & 1) ? r1 : r0;
                    uint32_t (&nx)[8] = (ps & 1) ? r0 : r1;
                    arrived(r);
                    if (ps < SCOLS / 8 - 1) ld(ps + 1, nx);
                    const float4 v0 = lds128(vj + 32 * ps), v1 = lds128(vj + 32 * ps + 16);
                    const float v[8] = {v0.x, v0.y, v0.z, v0.w, v1.x, v1.y, v1.z, v1.w};
#pragma unroll
                    for (int j = 0; j < 8; ++j) {
                        const float e = ex2(__uint_as_float(r[j]));
                        a[j & 3] = fmaf(e, v[j], a[j & 3]);
                        cs[ps * 8 + j] = fmaf(e, vi, cs[ps * 8 + j]);
                    }
                }
                sum = (a[0] + a[1]) + (a[2] + a[3]);
            }
            rowbuf[(s * SGRP + grp) * TM + row] = sum;
            // accumulator, stage (V_I has been read) and row sums of the tile
            fence_proxy_async();
            fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(&used[s]);
        }
        // column sums of the item: over the 32 rows of the warp, then the four
        // row quarters (fixed order)
        tcs_colsum64(cs, lane);
        *reinterpret_cast<float2*>(&colbuf[quarter * SN + grp * SCOLS + 2 * lane]) =
            make_float2(cs[0], cs[1]);
    }
    if (fail) atomicExch(&s_fail, 1);
    fence_before();
    __syncthreads();
    fence_after();
    if (threadIdx.x < SN)
        pcol[(size_t)blockIdx.x * SN + threadIdx.x] =
            ((colbuf[threadIdx.x] + colbuf[SN + threadIdx.x]) + colbuf[2 * SN + threadIdx.x]) +
            colbuf[3 * SN + threadIdx.x];
    if (threadIdx.x == 0 && s_fail) atomicExch(err, 1);
    if (warp == SEPI_TCS + 1) {
        __syncwarp();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem),
                     "r"(2 * SN));
    }
}

// O = noise V + the row partials of the point's tile a (pairs (a, J), J >= a,
// one each) + the column partials of the work items of column tile a, in a
// fixed order, rounded to FP32.  A CTA takes the 128 rows of one tile, eight groups
// of threads every eighth partial each, with TwoSum on FP32 pairs (2^-47; two FP64
// additions per clock and SM made the FP64 sum of all partials 0.25 of the product's
// 0.82 ms at n = 65536; this takes 0.02 ms), the groups' sums in FP64.  Where an infinity or
// an overflow on the way has spoilt a pair, the group's partials are added in FP64.
__global__ void __launch_bounds__(1024)
    tcs_reduce_kernel(const float* __restrict__ prow, const float* __restrict__ pcol,
                      const int* __restrict__ col_start, const int* __restrict__ col_items,
                      int64_t n_t, const float* __restrict__ V, float noise,
                      float* __restrict__ O, int64_t n) {
    __shared__ double red[8][TM];
    const int64_t a = blockIdx.x;
    const int r = threadIdx.x & (TM - 1), g = threadIdx.x / TM;
    float s = 0.f, c = 0.f;
    auto each = [&](auto&& add) {
#pragma unroll 4
        for (int64_t J = a / 2 + g; J < (n_t + 1) / 2; J += 8) add(prow[tcs_pair(J, a) * TM + r]);
#pragma unroll 4
        for (int e = col_start[a / 2] + g; e < col_start[a / 2 + 1]; e += 8)
            add(pcol[(size_t)col_items[e] * SN + (a & 1) * TN + r]);
    };
    each([&](float x) {
        const float t = s + x;
        const float z = t - s;
        c += (s - (t - z)) + (x - z);
        s = t;
    });
    double sum = (double)s + (double)c;
    if (!isfinite(sum)) {
        sum = 0.0;
        each([&](float x) { sum += (double)x; });
    }
    red[g][r] = sum;
    __syncthreads();
    const int64_t i = a * TM + r;
    if (g != 0 || i >= n) return;
    double o = (double)noise * (double)V[i];
#pragma unroll
    for (int q = 0; q < 8; ++q) o += red[q][r];
    O[i] = (float)o;
}

// V column k as FP32, zero past n (the ring's V_I and the resident V_J).
__global__ void tcs_stage_v_kernel(const float* __restrict__ V, int64_t n, int64_t n_pad,
                                   float* __restrict__ Vs) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n_pad;
         i += (int64_t)gridDim.x * blockDim.x)
        Vs[i] = (i < n) ? V[i] : 0.f;
}

template <int KCH>
void launch_tcs(const Ctx& h, const float* Vs, float* prow, float* pcol, cudaStream_t st) {
    using S = TcsSmem<KCH>;
    allow_smem(kv_tcs_kernel<KCH>, S::kTotal);
    const uint64_t wait_ns = h.opt.wait_limit_ns > 0 ? (uint64_t)h.opt.wait_limit_ns : kWaitNs;
    kv_tcs_kernel<KCH><<<(unsigned)h.tcs_nitems, SWARPS_TCS * 32, S::kTotal, st>>>(
        reinterpret_cast<const __nv_bfloat16*>(h.tcA.p),
        reinterpret_cast<const __nv_bfloat16*>(h.tcB.p), Vs, (h.n + TM - 1) / TM,
        reinterpret_cast<const int4*>(h.tcs_work.p), prow, pcol, h.tc_err.p, wait_ns,
        h.opt.wait_stall ? 1 : 0);
    KPCG_LAUNCHED("kv_tcs_kernel");
}

// Work items for n_t tiles of 128: column tile J (256) takes the row tiles 0..2J+1 in
// runs of at most G, launched longest first; the items of each column tile are listed (CSR) for the reduction.
void tcs_plan(Ctx& h, int64_t n_t) {
    if (h.tcs_n == h.n) return;
    const int sms = sm_count_tc();
    // G: whole waves of items (one per SM), an item costing its tiles plus about
    // eight more for its start and end.  (At least 16 tiles per item left 104 of 152
    // SMs idle at n = 4096: 0.069 ms per product against 0.052 ms.)
    const int64_t n_c = (n_t + 1) / 2;  // column tiles of 256
    int G = 1;
    double best = 1e300;
    for (int g = 1; g <= 128; ++g) {
        double cnt = 0.0;
        for (int64_t J = 0; J < n_c; ++J) cnt += (double)((std::min(2 * J + 2, n_t) + g - 1) / g);
        const double cost = std::ceil(cnt / sms) * (g + 8.0);
        if (cost < best * 0.999) {
            best = cost;
            G = g;
        }
    }
    std::vector<int4> items;
    for (int64_t J = 0; J < n_c; ++J) {
        const int64_t rows = std::min(2 * J + 2, n_t);
        for (int64_t I = 0; I < rows; I += G)
            items.push_back(make_int4((int)J, (int)I, (int)std::min<int64_t>(I + G, rows), 0));
    }
    std::stable_sort(items.begin(), items.end(),
                     [](const int4& a, const int4& b) { return (a.z - a.y) > (b.z - b.y); });
    std::vector<int> cols((size_t)n_c + 1 + items.size(), 0);
    for (const int4& it : items) ++cols[(size_t)it.x + 1];
    for (int64_t J = 0; J < n_c; ++J) cols[(size_t)J + 1] += cols[(size_t)J];
    std::vector<int> fill(cols.begin(), cols.begin() + n_c);
    for (size_t e = 0; e < items.size(); ++e)
        cols[(size_t)n_c + 1 + (size_t)fill[(size_t)items[e].x]++] = (int)e;
    int* w = h.tcs_work.need(items.size() * 4);
    int* c = h.tcs_cols.need(cols.size());
    KPCG_CUDA(cudaMemcpyAsync(w, items.data(), sizeof(int4) * items.size(), cudaMemcpyHostToDevice,
                              h.stream));
    KPCG_CUDA(cudaMemcpyAsync(c, cols.data(), sizeof(int) * cols.size(), cudaMemcpyHostToDevice,
                              h.stream));
    KPCG_CUDA(cudaStreamSynchronize(h.stream));
    h.tcs_nitems = (int)items.size();
    h.tcs_n = h.n;
}

}  // namespace

// Usable while n_t (n_t + 1) x 128 FP32 values stay within 4 GiB, i.e. up to
// n ~ 370 000 (its row partials are about a quarter of that); beyond that the
// one-sided kernel evaluates every entry.
bool kv_tcs_usable(const Ctx& h) {
    const double n_t = (double)((h.n + TM - 1) / TM);
    const double bytes = n_t * (n_t + 1.0) / 2.0 * 2.0 * TM * 4.0;
    return h.n > TM && kv_tc_supported(h.d) && bytes <= 4.0 * 1024 * 1024 * 1024;
}

void kv_tcs_apply(Ctx& h, const float* V, int64_t ldv, int c, float* O, int64_t ldo,
                  float noise) {
    if (h.n <= 0 || c <= 0) return;
    cudaStream_t st = h.stream;
    const int64_t n = h.n;
    const int64_t n_pad = ((n + TM - 1) / TM) * TM;
    const int64_t n_t = n_pad / TM;
    tc_prepare(h);  // the BF16x3 operands of kv_tc.cu (and its error flag)
    const int kch = h.tc_kch;
    tcs_plan(h, n_t);
    float* Vs = h.tcsV.need((size_t)n_pad);
    float* prow = h.tcsRow.need((size_t)tcs_pair((n_t + 1) / 2, 0) * TM);
    float* pcol = h.tcsCol.need((size_t)h.tcs_nitems * SN);
    const int* cols = h.tcs_cols.p;
    for (int k = 0; k < c; ++k) {
        tcs_stage_v_kernel<<<(unsigned)std::min<int64_t>((n_pad + 255) / 256, 2048), 256, 0, st>>>(
            V + (int64_t)k * ldv, n, n_pad, Vs);
        KPCG_LAUNCHED("tcs_stage_v_kernel");
        if (kch == 1)
            launch_tcs<1>(h, Vs, prow, pcol, st);
        else
            launch_tcs<2>(h, Vs, prow, pcol, st);
        tcs_reduce_kernel<<<(unsigned)n_t, 1024, 0, st>>>(
            prow, pcol, cols, cols + (n_t + 1) / 2 + 1, n_t, V + (int64_t)k * ldv, noise,
            O + (int64_t)k * ldo, n);
        KPCG_LAUNCHED("tcs_reduce_kernel");
    }
}

}  // namespace kpcg

// K_UX K_XU of the Nystrom set-up (Sec. 3.1) in fixed point on the tensor cores.
//
// M = noise K_UU + K_UX K_XU is nearly singular (kappa ~ 1e11 at noise 1e-4) and the
// preconditioner it defines implicitly inverts K_UU, whose small eigenvalues are far below
// the 2^-48 relative error of a compensated-FP32 sum divided by the noise: such errors
// made the preconditioner indefinite and doubled the PCG iteration count.  So the sum
// needs FP64 accuracy, but n m^2 / 2 FP64 multiply-adds at two per clock and SM were most
// of the set-up.  Here the entries of K_XU (FP32 pairs, 48 bits) are
// cut into eight balanced bytes, k = S sum_a d_a 2^(-7-8a), a = 0..7, S a power of
// two >= 2 max|k|, exact in FP16, and
//     (K_UX K_XU)_ab = S^2 sum_l 2^(-14-8l) L_l,  L_l = sum_{p+q=l} sum_i d_p(i,a) d_q(i,b),
// l = 0..7, each L_l an MMA chain whose FP32 accumulator holds an integer: |d_0| <= 65,
// the others <= 128, so over 128 rows |L_l| < 7.1 x 128 x 2^14 < 2^24.  After every 128
// rows the levels go into two 64-bit integers per entry (l = 0..3 and 4..7), at the end of
// a work item to FP64.  What is lost: an entry's digits below 2^-63 S and the levels >= 8
// (about 2^-64 S^2 per row, of either sign); the sum itself has no rounding.  On the
// diagonal the squares d_4(i,a)^2 of level 8 are of one sign, 2^-66 S^2 per row, and made a
// narrow kernel's entries at n = 65536 up to 1.3e-14 too small (FP64 sums: 2e-16 .. 2e-15):
// the digits' kernel adds them up beside its work and they go into the sum (6e-17).  With
// seven digits the levels lost would be 2^-56 S^2 per row, more than the rounding of an
// FP64 sum.
//
// Layout.  syrk_digits_kernel lays the digits of a block of rows out as swizzled K-major
// operands: per 32 rows and 128 columns of K_XU four sub-tiles of 128 x 128 bytes, two
// digits x 32 rows each.  The block is sized to stay in L2 (96 MB of 129).  A work item is a
// 128 x 64 tile of the lower triangle of M over a range of the block's rows; the 64
// columns of the second operand are half of a column tile.  10 warps: warp 0
// bulk-copies 32 rows per ring stage, warp 1 issues the 72 MMAs of a stage (36 digit pairs x
// K = 32), 8 epilogue warps read the levels after four stages.
// TMEM: 8 levels x 64 columns, all of it.  Every wait is bounded.
//
// What bounds it: the MMAs, 64 cycles each with A in shared memory (N = 64 needs 32), and
// the levels' readings, which they don't overlap (the levels fill TMEM).  Against the FP64
// kernel it replaces (64 x 64 tiles of DFMAs), with digits and maximum: n = 65536,
// m = 1024 3.3 ms (68), n = 20000, m = 1024 1.03 ms (22.3), m = 256 0.14 ms (1.5), n = 1030,
// m = 200 0.038 ms (0.18), n = 300, m = 32 0.034 ms (0.094), n = 1 0.032 ms (0.022): the
// three launches.  Relative error of the sum against quad precision 5e-17 .. 4e-16
// (FP64: 1e-16 .. 2e-15).
#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>

#include "precond.cuh"
#include "tcgen05.cuh"

namespace kpcg {
namespace {

constexpr int YND = 8;             // digits, levels
constexpr int YN = 64;             // columns of the second operand
constexpr int YR = 32;             // rows per stage
constexpr int YG = 4;              // stages between two readings of the levels
constexpr int YNST = 2;            // ring depth
constexpr int YEPI = 8;            // epilogue warps
constexpr int YWARPS = 2 + YEPI;
constexpr uint32_t kSubA = 128 * 128;      // sub-tile: 128 columns of K_XU x 128 bytes
constexpr uint32_t kTileA = 4 * kSubA;     // two digits per sub-tile
constexpr uint32_t kTileB = kTileA / 2;
constexpr uint32_t kStageY = kTileA + kTileB;
constexpr uint32_t kSmemY = 1024 + YNST * kStageY + 1024;
constexpr uint32_t kIdescY =
    (1u << 4) | ((uint32_t)(YN >> 3) << 17) | ((uint32_t)(128 >> 4) << 24);  // FP16, M = 128

// max |hi| over the pairs (bits of a non-negative float; NaN above infinity).
__global__ void pair_absmax_kernel(const float2* __restrict__ K, int64_t cnt,
                                   unsigned* __restrict__ out) {
    unsigned m = 0;
    for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < cnt;
         e += (int64_t)gridDim.x * blockDim.x) {
        const unsigned b = __float_as_uint(K[e].x) & 0x7fffffffu;
        m = b > m ? b : m;
    }
    m = __reduce_max_sync(0xffffffffu, m);
    if ((threadIdx.x & 31) == 0 && m) atomicMax(out, m);
}

// e with |k| <= 2^(e-1) for all entries k = hi + lo, up to the rounding in hi.  At
// least -100, where the last digit is below the smallest FP32 number.
__device__ __forceinline__ int pair_exponent(unsigned mx) {
    return max((int)(mx >> 23) - 125, -100);
}

// Digits of rows i0 .. i0 + nrows - 1 (zero past n and past column m), and the squares of
// the fifth added to sq, per column.  One thread per column and 8 rows.
__global__ void syrk_digits_kernel(const float2* __restrict__ KXU, int64_t n, int64_t m, int64_t i0,
                                   int64_t nrows, int64_t ct, int cw, const unsigned* __restrict__ mx,
                                   uint8_t* __restrict__ dig, unsigned long long* __restrict__ sq) {
    const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int64_t cols = ct * cw;
    if (e >= nrows / 8 * cols) return;
    const int64_t a = e % cols, r8 = e / cols;  // consecutive threads: consecutive columns
    // 2^(7 - exponent) from its bits: the products below and the epilogue's way back
    // rely on an exact power of two, exp2f promises two ulps.  The exponent is -100 .. 130.
    const float sc = __int_as_float((127 + 7 - pair_exponent(*mx)) << 23);
    float h[8], l[8];
#pragma unroll
    for (int r = 0; r < 8; ++r) {
        const int64_t i = i0 + r8 * 8 + r;
        const float2 k = (i < n && a < m) ? KXU[i * m + a] : make_float2(0.f, 0.f);
        h[r] = k.x * sc;
        l[r] = k.y * sc;
    }
    const int64_t chunk = r8 / 4;      // 32 rows
    const int c8 = (int)(r8 & 3);      // 16-byte chunk of the 64 bytes of a digit
    const int row = (int)(a & 127);
    const uint32_t sub = (uint32_t)cw * 128;
    uint8_t* base = dig + ((size_t)chunk * ct + (size_t)(a >> 7)) * 4 * sub + row * 128;
    float sum4 = 0.f;  // at most 8 x 2^14
#pragma unroll
    for (int d = 0; d < YND; ++d) {
        uint32_t w[4];
#pragma unroll
        for (int r = 0; r < 8; r += 2) {
            float v[2];
#pragma unroll
            for (int z = 0; z < 2; ++z) {
                // the digit of h + l; what is left is exact (TwoSum; s - v is exact)
                const float s = h[r + z] + l[r + z];
                const float bb = s - h[r + z];
                const float e = (h[r + z] - (s - bb)) + (l[r + z] - bb);
                v[z] = rintf(s);
                if (d == YND / 2) sum4 = fmaf(v[z], v[z], sum4);
                h[r + z] = (s - v[z]) * 256.f;
                l[r + z] = e * 256.f;
            }
            const __half2 p = __floats2half2_rn(v[0], v[1]);
            w[r >> 1] = *reinterpret_cast<const uint32_t*>(&p);
        }
        const int c = (d & 1) * 4 + c8;
        *reinterpret_cast<uint4*>(base + (size_t)(d >> 1) * sub + ((c ^ (row & 7)) * 16)) =
            make_uint4(w[0], w[1], w[2], w[3]);
    }
    if (sum4 > 0.f) atomicAdd(&sq[a], (unsigned long long)sum4);
}

// Tile x of the lower triangle: rows 128 T .. + 127, columns 64 u .. + 63, u < 2 T + 2.
__host__ __device__ inline void syrk_tile(int x, int& T, int& u) {
    T = 0;
    while ((T + 1) * (T + 2) <= x) ++T;
    u = x - T * (T + 1);
}

__global__ void __launch_bounds__(YWARPS * 32, 1)
    syrk_fx_kernel(const uint8_t* __restrict__ dig, int64_t m, int ct, int cw, int ngroups,
                   int groups_per_split, const unsigned* __restrict__ mx,
                   const unsigned long long* __restrict__ sq, int first, double* __restrict__ part, int* __restrict__ err, uint64_t wait_ns, int stall) {
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = reinterpret_cast<uint8_t*>(
        (reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    uint64_t* bars = reinterpret_cast<uint64_t*>(smem + YNST * kStageY);
    uint64_t* full = bars;           // [YNST] copies landed
    uint64_t* empty = full + YNST;   // [YNST] MMAs of the stage done
    uint64_t* lfull = empty + YNST;  // levels of YG stages ready
    uint64_t* lfree = lfull + 1;     // levels read
    uint64_t* done = lfree + 1;
    uint64_t* never = done + 1;  // test hook: no thread ever arrives here
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(never + 1);
    __shared__ int s_fail;

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    int T, u;
    syrk_tile((int)blockIdx.x, T, u);
    const int g0 = (int)blockIdx.y * groups_per_split;
    const int ng = max(0, min(ngroups - g0, groups_per_split));
    const int nst = ng * YG;

    if (threadIdx.x == 0) {
        for (int s = 0; s < YNST; ++s) {
            mbar_init(&full[s], 1);
            mbar_init(&empty[s], 1);
        }
        mbar_init(lfull, 1);
        mbar_init(lfree, YEPI);
        mbar_init(done, 1);
        mbar_init(never, 1);
        s_fail = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 1) {
        asm volatile(
            "tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                su32(tmem_slot)),
            "r"(512));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    fence_before();
    __syncthreads();
    fence_after();
    const uint32_t tmem = *tmem_slot;
    const uint64_t deadline = gtimer() + wait_ns;
    int fail = 0;

    if (warp == 0) {
        if (lane == 0) {
            int t = 0;
            for (; t < nst; ++t) {
                const int s = t % YNST;
                if (!mbar_wait_idle(&empty[s], ((uint32_t)(t / YNST) & 1u) ^ 1u, deadline)) {
                    fail = 1;
                    break;
                }
                uint8_t* st = smem + (size_t)s * kStageY;
                const uint32_t sub = (uint32_t)cw * 128;
                const uint8_t* row = dig + (size_t)(g0 * YG + t) * ct * 4 * sub;
                // columns 64 u .. + 63: half of every sub-tile of column tile u / 2
                const uint32_t half = (uint32_t)(u & 1) * (kSubA / 2);
                const uint32_t nb = min(kSubA / 2, sub - half);
                mbar_expect_tx(&full[s], 4 * (sub + nb));
                for (int q = 0; q < 4; ++q) {
                    bulk_g2s(st + q * kSubA, row + ((size_t)T * 4 + q) * sub, sub, &full[s]);
                    bulk_g2s(st + kTileA + q * (kSubA / 2), row + ((size_t)(u >> 1) * 4 + q) * sub + half,
                             nb, &full[s]);
                }
            }
            // the CTA exits only once the copies it issued have landed
            const uint64_t dl2 = gtimer() + 200000000ull;
            for (int q = (t > YNST ? t - YNST : 0); q < t; ++q)
                (void)mbar_wait(&full[q % YNST], (uint32_t)(q / YNST) & 1u, dl2);
        }
    } else if (warp == 1) {
        const uint32_t el = elect_one();
        // test hook: a wait on a barrier nothing arrives at runs out
        if (stall && !mbar_wait_warp(never, 0, deadline)) fail = 1;
        for (int t = 0; t < nst && !fail; ++t) {
            const int s = t % YNST, g = t / YG;
            if (!mbar_wait_warp(&full[s], (uint32_t)(t / YNST) & 1u, deadline) ||
                (t % YG == 0 && !mbar_wait_warp(lfree, ((uint32_t)g & 1u) ^ 1u, deadline))) {
                fail = 1;
                break;
            }
            fence_after();
            const uint32_t a0 = su32(smem + (size_t)s * kStageY), b0 = a0 + kTileA;
#pragma unroll
            for (int z = 0; z < 2; ++z)
#pragma unroll
                for (int p = 0; p < YND; ++p)
#pragma unroll
                    for (int q = 0; q < YND - p; ++q)  // neighbours in different levels
                        mma_ss(tmem + (uint32_t)((p + q) * YN),
                               sdesc(a0 + (uint32_t)(p >> 1) * kSubA + (uint32_t)((p & 1) * 64 + z * 32)),
                               sdesc(b0 + (uint32_t)(q >> 1) * (kSubA / 2) +
                                     (uint32_t)((q & 1) * 64 + z * 32)),
                               kIdescY, ((t % YG) | z | p) ? 1u : 0u, el);
            mma_commit(&empty[s], el);
            if (t % YG == YG - 1) mma_commit(lfull, el);
        }
        mma_commit(done, el);
        if (!mbar_wait_warp(done, 0, gtimer() + kWaitNs)) fail = 1;
    } else {
        const int quarter = warp & 3, half = (warp - 2) >> 2;
        const uint32_t base =
            tmem + ((uint32_t)(quarter * 32) << 16) + (uint32_t)(half * (YN / 2));
        long long hi[YN / 2], lo[YN / 2];  // levels 0..3 in units of the fourth, 4..7 of the last
#pragma unroll
        for (int b = 0; b < YN / 2; ++b) hi[b] = lo[b] = 0;
        for (int g = 0; g < ng; ++g) {
            if (!mbar_wait_warp(lfull, (uint32_t)g & 1u, deadline)) {
                fail = 1;
                break;
            }
            fence_after();
#pragma unroll
            for (int b = 0; b < YN / 2; b += 4) {
                uint32_t r[YND][4];
#pragma unroll
                for (int k = 0; k < YND; ++k)
                    asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0, %1, %2, %3}, [%4];"
                                 : "=r"(r[k][0]), "=r"(r[k][1]), "=r"(r[k][2]), "=r"(r[k][3])
                                 : "r"(base + (uint32_t)(k * YN + b)));
                tmem_wait_ld();
#pragma unroll
                for (int k = 0; k < YND; ++k)
                    asm volatile("" : "+r"(r[k][0]), "+r"(r[k][1]), "+r"(r[k][2]), "+r"(r[k][3])
                                 : : "memory");
                if (b + 4 == YN / 2) {
                    fence_before();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(lfree);
                }
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    int L[YND];
#pragma unroll
                    for (int k = 0; k < YND; ++k) L[k] = __float2int_rn(__uint_as_float(r[k][q]));
                    hi[b + q] += (long long)L[0] * 16777216 + (long long)L[1] * 65536 +
                                 (long long)L[2] * 256 + L[3];
                    lo[b + q] += (long long)L[4] * 16777216 + (long long)L[5] * 65536 +
                                 (long long)L[6] * 256 + L[7];
                }
            }
        }
        const int64_t a = (int64_t)T * 128 + quarter * 32 + lane;
        const int64_t b0 = (int64_t)u * YN + half * (YN / 2);
        const unsigned bits = *mx;
        const double sc = bits < 0x7f800000u ? ldexp(1.0, 2 * pair_exponent(bits))
                                             : __longlong_as_double(0x7ff8000000000000ll);
        double* P = part + (size_t)blockIdx.y * m * m;
        if (a < m)
#pragma unroll
            for (int b = 0; b < YN / 2; ++b) {
                if (b0 + b > a) continue;
                double v = fma((double)hi[b], 0x1p-38, (double)lo[b] * 0x1p-70) * sc;
                if (b0 + b == a && sq && blockIdx.y == 0) v = fma((double)sq[a], 0x1p-78 * sc, v);
                P[a * m + b0 + b] = first ? v : P[a * m + b0 + b] + v;
            }
    }
    if (fail) atomicExch(&s_fail, 1);
    fence_before();
    __syncthreads();
    fence_after();
    if (threadIdx.x == 0 && s_fail) atomicExch(err, 1);
    if (warp == 1) {
        __syncwarp();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512));
    }
}

int sms_y() {
    static int cached = 0;
    if (!cached) {
        int dev = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&cached, cudaDevAttrMultiProcessorCount, dev);
        if (cached <= 0) cached = 152;
    }
    return cached;
}

}  // namespace

// Rows per block of digits and splits of its rows.
static void syrk_fx_plan(int64_t n, int64_t m, int64_t& rows, int& nsplit) {
    const int64_t ct = (m + 127) / 128, group = YR * YG;
    const int64_t want = std::max<int64_t>(group, (96ll << 20) / (ct * (int64_t)kTileA / YR));
    const int64_t groups = (n + group - 1) / group;
    const int64_t nblk = (groups * group + want - 1) / want;
    rows = (groups + nblk - 1) / nblk * group;
    const int64_t ub = (m + YN - 1) / YN;
    int64_t tiles = 0;
    for (int64_t T = 0; T < ct; ++T) tiles += std::min(2 * T + 2, ub);
    nsplit = (int)std::max<int64_t>(1, std::min<int64_t>(rows / group, sms_y() / tiles));
}

int syrk_fx_splits(int64_t n, int64_t m) {
    int64_t rows;
    int nsplit;
    syrk_fx_plan(n, m, rows, nsplit);
    return nsplit;
}

// What the work area holds before the digits: the largest entry, the flag of an expired wait,
// the squares of the fifth digits.
static size_t syrk_fx_head(int64_t m) {
    return 256 + sizeof(unsigned long long) * (size_t)((m + 127) / 128 * 128);
}

// Columns a column tile has in memory: up to 128 the eights that hold m.  What the tiles
// in shared memory keep past them reaches only rows and columns of the sum past m, which are
// not stored.  (With 128 of them a set-up of n = 1030, m = 8 worked on 2.4 MB instead of
// 0.15, and the driver's calls for more than 2 MB are slow: 314 -> 167 us.)
static int syrk_fx_cols(int64_t m) { return m > 120 ? 128 : (int)((m + 7) / 8 * 8); }

size_t syrk_fx_bytes(int64_t n, int64_t m) {
    int64_t rows;
    int nsplit;
    syrk_fx_plan(n, m, rows, nsplit);
    return syrk_fx_head(m) +
           (size_t)(rows / YR) * (size_t)((m + 127) / 128) * (size_t)syrk_fx_cols(m) * 512;
}

const int* syrk_fx(const float2* KXU, int64_t n, int64_t m, uint8_t* work, double* part,
                   int64_t stall_ns, cudaStream_t st) {
    const int64_t ct = (m + 127) / 128, group = YR * YG;
    const int cw = syrk_fx_cols(m);
    int64_t rows;
    int nsplit;
    syrk_fx_plan(n, m, rows, nsplit);
    const int64_t ub = (m + YN - 1) / YN;
    int tiles = 0;
    for (int64_t T = 0; T < ct; ++T) tiles += (int)std::min(2 * T + 2, ub);
    const size_t head = syrk_fx_head(m);
    unsigned* mx = reinterpret_cast<unsigned*>(work);
    int* err = reinterpret_cast<int*>(work + 128);
    unsigned long long* sq = reinterpret_cast<unsigned long long*>(work + 256);
    uint8_t* dig = work + head;
    KPCG_CUDA(cudaMemsetAsync(work, 0, head, st));
    pair_absmax_kernel<<<(unsigned)std::min<int64_t>((n * m + 1023) / 1024, 152 * 8), 256, 0, st>>>(
        KXU, n * m, mx);
    KPCG_LAUNCHED("pair_absmax_kernel");
    allow_smem(syrk_fx_kernel, kSmemY);
    for (int64_t i0 = 0; i0 < n; i0 += rows) {
        const int64_t here = std::min(rows, (n - i0 + group - 1) / group * group);
        const int64_t thr = here / 8 * ct * cw;
        syrk_digits_kernel<<<(unsigned)((thr + 255) / 256), 256, 0, st>>>(KXU, n, m, i0, here, ct, cw, mx,
                                                                          dig, sq);
        KPCG_LAUNCHED("syrk_digits_kernel");
        const int ngroups = (int)(here / group);
        // every split writes (the first block) or adds to its part, also when it has no rows
        syrk_fx_kernel<<<dim3((unsigned)tiles, (unsigned)nsplit), YWARPS * 32, kSmemY, st>>>(
            dig, m, (int)ct, cw, ngroups, (ngroups + nsplit - 1) / nsplit, mx,
            i0 + rows >= n ? sq : nullptr, i0 == 0, part, err,
            stall_ns > 0 ? (uint64_t)stall_ns : kWaitNs, stall_ns > 0 ? 1 : 0);
        KPCG_LAUNCHED("syrk_fx_kernel");
    }
    return err;
}

}  // namespace kpcg

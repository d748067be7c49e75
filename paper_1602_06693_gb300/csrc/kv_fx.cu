// FP64-class K.V in fixed point on the tensor cores (sm_103a), d <= 16.
//
// O = K V + noise V (or B - that), K_ij = s^2 2^(-|y_i - y_j|^2) (Eq. 1 with
// y = x' sqrt(log2 e)), V and O in FP64, entries rebuilt per tile (the
// matrix-free product of Sec. 2.1).  GB300 issues two FP64 operations per
// clock and SM, so an entry whose distance, exp and products run on that pipe
// costs about 28 x 64 issue slots of the FP32 pipe.  Here none of them does:
//
// 1. Distance.  y / S (S a power of two >= max(2, |y|)) is cut into six balanced
//    10-bit integer slices, y = S 2^-9 sum_a s_a 2^(-10a), exact in FP16.
//    Level k of y_i.y_j is L_k = sum_{a+b=k} sum_r s_a(i,r) s_b(j,r), a chain of
//    FP16 MMAs whose FP32 accumulator holds an integer: |L_k| <= (k+1) d 2^18,
//    at most 2^24 and so exact for every level at d <= 10 and for levels 0..3 at
//    d <= 16 (above that only the last two levels can round, by one unit of
//    2^(-57) S^2 or less).  -|y_i|^2 / 2 and -|y_j|^2 / 2, from the same slices and
//    levels in 128-bit integers, ride along as digits in four spare K columns,
//    so the six accumulators hold -|y_i - y_j|^2 / 2 in units of S^2 2^(-18-10k).
//    Levels >= 6 of y_i.y_j are dropped: ~2^-59 S^2 of the exponent, independent
//    per entry, of no sign.  (They are kept in |y|^2: its dropped part would be
//    positive, a bias of 2^-57 S^2 common to a point's entries; and the
//    entry of a point with itself, where it would not cancel, is set to s^2.)
// 2. exp2 (after P. T. P. Tang's table-driven method, 1989).  The exponent is -n/4096 + r,
//    |r| <= 2^-13, r = rh + rl in FP32 without rounding of the leading levels;
//    2^r - 1 by its Taylor polynomial to r^3 with the linear part in two FP32
//    numbers; T = 2^(-(n mod 4096)/4096) is a 57-bit integer of the table, the
//    product T (2^r - 1) two FP32 numbers whose integer parts are read off the
//    mantissas of sums with 1.5 2^k and added to T as 64-bit integers; the
//    result is shifted right by n >> 12 and rounded.  K/s^2 = M 2^-62, M an integer,
//    to about 2^-54 relative and 2^-63 absolute.
// 3. Contraction.  M is written in eight balanced digits of base 256: 128 is added to
//    all of its bytes but the top one, and what the 128s put into a sum, which depends on
//    V alone, is taken out of the integer sums again.  The bytes are FP16 subnormals as
//    they stand (byte 2^-24), written to tensor memory as the A operand of a second chain of
//    MMAs against V cut into eight balanced bytes per column (scaled by a
//    power of two per column).  Products of byte levels l = a + b add in FP32
//    accumulators that hold integers below 2^24 over 64 columns; they are then
//    added to 32-bit integers, which go to FP64 once per work item.  Levels
//    >= 8 are dropped: 2^-62 of max|K| max|V| per product or less, of either sign.  The
//    sum itself has no rounding.
//
// Entries and columns of V are thus cut at an absolute place, 2^-63 of the largest.  On n
// entries that are small against one (a narrow kernel, V of one sign) such errors add up
// unless they are of either sign: with seven unsigned bytes (unit 2^-55) a row of n = 65536
// was off by 2e-14, with eight unsigned ones, for a constant V with digits, by 1.4e-14
// (products of its constant digits with unsigned bytes in the dropped levels), with these by
// 7e-16; FP64 sums by 1e-15 to 3e-15.
//
// What bounds it: issue of the epilogue, 84 instructions per entry with one
// column (ncu at n = 16384: issue 73%, the ALU pipe 43%, FP32 39%, DRAM the operands once),
// nearly independent of the number of columns, where the FP64 kernel needs 28 + 2 c FP64
// operations per pair of points (two per clock and SM) and the double-float one 67 + 25 c
// FP32 instructions.  n = 65536, d = 8: 12.9 ms with one column (FP64: 119.6 ms; 12.1 ms with
// seven unsigned bytes); n = 45730, d = 9, 17 columns: 8.7 ms (double-float: 36.1 ms).
// Errors against extended precision on random, constant and smooth vectors: 1e-16 to
// 5e-16 of the result.
//
// Layout.  A work item is 128 rows x a run of 64-column groups of two 32-column
// units.  18 warps: warp 0 bulk-copies a group's B operand and V bytes into a
// ring, warp 1 issues all MMAs from one thread, 16 epilogue warps (four row
// quarters, the TMEM lanes a warp may read, x four groups of 8 columns of a
// unit).  Every TMEM buffer is single: the levels of a unit are read into
// registers at once and their buffer handed back, so the distance MMAs of the
// next unit and the byte MMAs of the last one run behind a unit's evaluation.
// All bytes of K accumulate into the same columns [level l][column of V], byte a
// against V's bytes moved down by a levels (operand rows that start a x cpad rows
// earlier, in zeros), so that one accumulator takes all of them: the order of MMAs whose
// accumulators overlap without being the same is not defined.  (Units of 16 columns with
// two sets of warps on alternate units took a third longer: twice the distance MMAs, and an
// MMA takes the same time whatever N is below 64.)
// TMEM: 6 x 32 columns of levels, 8 x 16 of bytes, 8 x cpad (<= 192) of sums: all of it.
// Every mbarrier wait is bounded.
#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstddef>
#include <cstring>
#include <vector>

#include "ctx.cuh"
#include "tcgen05.cuh"

namespace kpcg {
namespace {

constexpr int QNS = 6;       // slices of y, levels of the distance
constexpr int QU = 32;       // columns per unit (N of the distance MMAs)
constexpr int QG = 64;       // columns per group (one ring stage, one drain)
constexpr int QUG = QG / QU;  // units per group
constexpr int QNK = 8;       // bytes of K
constexpr int QNV = 8;       // bytes of V
constexpr int QEPI = 16;     // epilogue warps
constexpr int QWARPS = 2 + QEPI;
constexpr int QNST = 2;      // ring depth
constexpr int QTAB = 4096;   // table of 2^(-j/4096)
constexpr int QMAXC = 24;    // columns of V per pass
// TMEM columns of the levels (32 k), the bytes (16 a) and the sums (cpad l + column)
constexpr uint32_t kLevT = 0, kByteT = QNS * QU, kSumT = kByteT + QNK * QU / 2;
// 64-column groups per work item at most: the 32-bit sums take 2^24 per group
constexpr int kMaxGroups = 120;
// Columns of V with at most so many values that are not zero go entry by entry
constexpr int kFew = 32;
// What is known of a pass's columns of V; all but the lists is cleared before.
struct FxCols {
    unsigned long long mx[QMAXC];   // bits of max |v|
    unsigned long long nnz[QMAXC];  // values that are not zero
    unsigned got[QMAXC];            // entries of the lists
    int row[QMAXC][kFew];           // where nnz <= kFew: the values, in any order
    double val[QMAXC][kFew];
};

// Integer parts of the table correction: bits(M1) 2^21 + bits(M3) with
// M1 = 1.5 2^-12 (unit 2^-35) and M3 = 1.5 2^-33 (unit 2^-56), taken off the table's
// entries so that the mantissas can be added as they are.
constexpr uint64_t kTabOff = ((uint64_t)0x39C00000u << 21) + 0x2F400000u;
// 128 in every byte of an entry but the top one
constexpr uint64_t kDigitOff = 0x0080808080808080ull;

struct FxScale {
    float w0, w1, w2, w3, w4;  // S^2 2^(-17 - 10 k)
};

template <int SUBT, int CPAD>
struct FxSmem {
    static constexpr uint32_t kA = SUBT * 128 * 128;
    static constexpr uint32_t kB = SUBT * QU * 128;        // one unit
    static constexpr uint32_t kV = QNV * CPAD * 128;       // one group: rows (byte, column)
    static constexpr uint32_t kZ = (QNK - 1) * CPAD * 128; // rows of zeros in front of them
    static constexpr uint32_t kStage = QUG * kB + kZ + kV;
    static constexpr uint32_t kTab = QTAB * 8;
    static constexpr uint32_t kBars = 1024;  // and the V sums behind them
    static constexpr uint32_t kTotal = 1024 + kA + QNST * kStage + kTab + kBars;
    static_assert(256 + QNV * CPAD * 4 <= kBars, "barriers and V sums");
    static_assert(CPAD * 128 * 8 <= kA + QNST * kStage, "combination buffer");
};

// FP16 x FP16 -> FP32, K-major, M = 128
__device__ __forceinline__ constexpr uint32_t fx_idesc(int n) {
    return (1u << 4) | ((uint32_t)(n >> 3) << 17) | ((uint32_t)(128 >> 4) << 24);
}
__device__ __forceinline__ void tmem_ld4_nw(uint32_t taddr, uint32_t* r) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0, %1, %2, %3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"(taddr));
}
__device__ __forceinline__ void tmem_bind4(uint32_t* r) {
    asm volatile("" : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]) : : "memory");
}
__device__ __forceinline__ void tmem_ld2(uint32_t taddr, uint32_t* r) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x2.b32 {%0, %1}, [%2];"
                 : "=r"(r[0]), "=r"(r[1])
                 : "r"(taddr));
    asm volatile("tcgen05.wait::ld.sync.aligned;" : "+r"(r[0]), "+r"(r[1]) : : "memory");
}
__device__ __forceinline__ void tmem_st2(uint32_t taddr, uint32_t a, uint32_t b) {
    asm volatile("tcgen05.st.sync.aligned.32x32b.x2.b32 [%0], {%1, %2};" ::"r"(taddr), "r"(a),
                 "r"(b)
                 : "memory");
}
__device__ __forceinline__ uint32_t prmt(uint32_t a, uint32_t b, uint32_t sel) {
    return __byte_perm(a, b, sel);
}

// kDigitOff + M with K/s^2 = M 2^-62 from the six level accumulators of an entry (step 2
// of the file's comment); tab holds round(2^(56 - j/4096)) - kTabOff.
__device__ __forceinline__ uint64_t fx_entry(float L0, float L1, float L2, float L3, float L4,
                                             float L5, const FxScale& w,
                                             const uint64_t* __restrict__ tab) {
    const float a0 = __fmul_rn(L0, w.w0);
    float s = fmaf(L1, w.w1, a0);
    s = fmaf(L2, w.w2, s);
    s = fmaf(L3, w.w3, s);
    s = fmaxf(s, -1000.f);
    const float t = fmaf(s, -4096.f, 12582912.f);
    const uint32_t nb = __float_as_uint(t) - 0x4B400000u;  // n
    const float u = __fadd_rn(t, -12582912.f);
    // r = exponent + n / 4096: the leading levels cancel without rounding
    float b = fmaf(u, 0x1p-12f, a0);
    b = fmaf(L1, w.w1, b);
    b = fmaf(L2, w.w2, b);
    const float rh = fmaf(L3, w.w3, b);
    float rl = fmaf(L3, w.w3, __fsub_rn(b, rh));
    rl = fmaf(fmaf(L5, 0x1p-10f, L4), w.w4, rl);
    // eh + el = 2^(rh + rl) - 1
    constexpr float kC1h = 0x1.62e43p-1f, kC1l = -0x1.05c61p-29f;  // ln 2
    constexpr float kC2 = 0x1.ebfbep-3f, kC3 = 0x1.c6b08ep-5f;      // ln^2 2 / 2, ln^3 2 / 6
    const float p = __fmul_rn(rh, kC1h);
    float pl = fmaf(rh, kC1h, -p);
    pl = fmaf(rh, kC1l, pl);
    pl = fmaf(rl, fmaf(rh, 2.f * kC2, kC1h), pl);
    const float q = __fmul_rn(rh, fmaf(rh, kC3, kC2));
    const float eh = fmaf(rh, q, p);
    const float el = __fadd_rn(fmaf(rh, q, __fsub_rn(p, eh)), pl);
    // T = Tf + Tl from the table integer (hi: Tf in 24 bits, lo: the rest)
    const uint64_t T = tab[nb & (QTAB - 1)];
    const uint32_t thi = (uint32_t)(T >> 32), tlo = (uint32_t)T;
    const float Tf = __uint_as_float(thi + ((0x39C00000u >> 11) + 0x3E800000u));
    const float Tl = fmaf((float)tlo, 0x1p-56f, 0x1.7ap-27f);  // + 0x2F400000 2^-56
    const float ph = __fmul_rn(Tf, eh);
    float pt = fmaf(Tf, eh, -ph);
    pt = fmaf(Tf, el, pt);
    pt = fmaf(Tl, eh, pt);
    // (the last levels can cancel part of ph, so g1 takes the rounded sum: |y| < 2^-35)
    const float g1 = __fadd_rn(__fadd_rn(ph, pt), 0x1.8p-12f);
    const float y = __fadd_rn(__fsub_rn(ph, __fadd_rn(g1, -0x1.8p-12f)), pt);
    const float g3 = __fadd_rn(y, 0x1.8p-33f);
    uint64_t M = T + ((uint64_t)__float_as_uint(g1) << 21);
    M += (uint64_t)__float_as_uint(g3);
    // rounded to nearest: cut off instead, the 2^-63 lost on average by each of n
    // entries would add up on a vector of one sign
    uint64_t r;
    asm("shr.u64 %0, %1, %2;" : "=l"(r) : "l"(M << 7), "r"(nb >> 12));  // 0 from 64 on
    return (r + (2 * kDigitOff + 1)) >> 1;
}

// CU: columns of V whose sums are kept (<= CPAD)
template <int SUBT, int KS, int CPAD, int CU>
__global__ void __launch_bounds__(QWARPS * 32, 1)
    kv_fx_kernel(const __half* __restrict__ Aop, const __half* __restrict__ Bop,
                 const __half* __restrict__ Vop, const int* __restrict__ vsum, int64_t n,
                 int64_t n_pad, int ncols, int groups_per_split, FxScale w, const uint64_t* __restrict__ gtab,
                 double* __restrict__ part, int* __restrict__ err, uint64_t wait_ns, int stall) {
    using S = FxSmem<SUBT, CPAD>;
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = reinterpret_cast<uint8_t*>(
        (reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    uint8_t* sA = smem;
    uint8_t* sStage = smem + S::kA;
    uint64_t* tab = reinterpret_cast<uint64_t*>(sStage + QNST * S::kStage);
    uint64_t* bars = reinterpret_cast<uint64_t*>(sStage + QNST * S::kStage + S::kTab);
    uint64_t* full = bars;           // [QNST] bulk copies landed
    uint64_t* empty = bars + QNST;   // [QNST] MMAs of the group done
    uint64_t* tfull = empty + QNST;  // levels of a unit ready
    uint64_t* tempty = tfull + 1;    // levels of a unit in registers
    uint64_t* bfull = tempty + 1;    // bytes of a unit stored
    uint64_t* bfree = bfull + 1;     // byte MMAs of a unit done
    uint64_t* afull = bfree + 1;
    uint64_t* done = afull + 1;
    uint64_t* never = done + 1;  // test hook: no thread ever arrives here
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(never + 1);
    // 128 (V bytes above level l) over the item's columns: [l][column of V]
    int* off = reinterpret_cast<int*>(sStage + QNST * S::kStage + S::kTab + 256);
    double* comb = reinterpret_cast<double*>(smem);  // after the loop: [CPAD][128]
    __shared__ int s_fail;

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int64_t rt = blockIdx.x;
    const int64_t g0 = (int64_t)blockIdx.y * groups_per_split;
    const int ngroups = (int)max((int64_t)0, min(n_pad / QG - g0, (int64_t)groups_per_split));
    const int nunits = QUG * ngroups;

    for (int e = threadIdx.x; e < QTAB; e += blockDim.x) tab[e] = gtab[e];
    for (int e = threadIdx.x; e < QNST * (int)(S::kZ / 16); e += blockDim.x)
        *reinterpret_cast<uint4*>(sStage + (size_t)(e / (S::kZ / 16)) * S::kStage + QUG * S::kB +
                                  (e % (S::kZ / 16)) * 16) = make_uint4(0u, 0u, 0u, 0u);
    fence_proxy_async();
    if (threadIdx.x == 0) {
        for (int s = 0; s < QNST; ++s) {
            mbar_init(&full[s], 1);
            mbar_init(&empty[s], 1);
        }
        mbar_init(tfull, 1);
        mbar_init(tempty, QEPI);
        mbar_init(bfull, QEPI);
        mbar_init(bfree, 1);
        mbar_init(afull, 1);
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
    const int quarter = warp & 3;
    const int cg = (warp - 2) >> 2;  // columns 8 cg .. + 7 of a unit, levels 2 cg, 2 cg + 1 of a group
    const int row = quarter * 32 + lane;
    int acc[2][CU];  // the two levels' sums
#pragma unroll
    for (int k = 0; k < CU; ++k) acc[0][k] = acc[1][k] = 0;

    if (warp == 0) {
        if (lane == 0) {
            mbar_expect_tx(afull, S::kA);
            bulk_g2s(sA, reinterpret_cast<const uint8_t*>(Aop) + (size_t)rt * S::kA, S::kA, afull);
            int g = 0;
            for (; g < ngroups; ++g) {
                const int s = g % QNST;
                if (!mbar_wait(&empty[s], ((uint32_t)(g / QNST) & 1u) ^ 1u, deadline)) {
                    fail = 1;
                    break;
                }
                uint8_t* st = sStage + (size_t)s * S::kStage;
                mbar_expect_tx(&full[s], QUG * S::kB + S::kV);
                bulk_g2s(st, reinterpret_cast<const uint8_t*>(Bop) + (size_t)(g0 + g) * QUG * S::kB,
                         QUG * S::kB, &full[s]);
                bulk_g2s(st + QUG * S::kB + S::kZ,
                         reinterpret_cast<const uint8_t*>(Vop) + (size_t)(g0 + g) * S::kV, S::kV,
                         &full[s]);
            }
            // the CTA exits only once the copies it issued have landed
            const uint64_t dl2 = gtimer() + 200000000ull;
            for (int q = (g > QNST ? g - QNST : 0); q < g; ++q)
                (void)mbar_wait(&full[q % QNST], (uint32_t)(q / QNST) & 1u, dl2);
            (void)mbar_wait(afull, 0, dl2);
        }
        __syncwarp();
        int t[QNV * CPAD / 32];
#pragma unroll
        for (int e = 0; e < QNV * CPAD / 32; ++e) t[e] = 0;
        const int* vs = vsum + (size_t)g0 * (QNV * CPAD) + lane;
#pragma unroll 8
        for (int g = 0; g < ngroups; ++g)
#pragma unroll
            for (int e = 0; e < QNV * CPAD / 32; ++e) t[e] += __ldg(vs + (size_t)g * (QNV * CPAD) + e * 32);
#pragma unroll
        for (int e = 0; e < QNV * CPAD / 32; ++e) off[lane + e * 32] = t[e];
    } else if (warp == 1) {
        const uint32_t el = elect_one();
        // test hook: a wait on a barrier nothing arrives at runs out
        if (stall && !mbar_wait_warp(never, 0, deadline)) fail = 1;
        if (!fail && !mbar_wait_warp(afull, 0, deadline)) fail = 1;
        fence_after();
        const uint32_t a0 = su32(sA);
        // the levels of unit t
        auto level_mmas = [&](int t) -> bool {
            const int g = t / QUG, s = g % QNST;
            if ((t % QUG == 0 && !mbar_wait_warp(&full[s], (uint32_t)(g / QNST) & 1u, deadline)) ||
                !mbar_wait_warp(tempty, ((uint32_t)t & 1u) ^ 1u, deadline))
                return false;
            fence_after();
            const uint32_t b0 =
                su32(sStage + (size_t)s * S::kStage + (size_t)(t % QUG) * S::kB);
#pragma unroll
            for (int a = 0; a < QNS; ++a)
#pragma unroll
                for (int z = 0; z < KS; ++z)
#pragma unroll
                    for (int k = a; k < QNS; ++k) {  // neighbours in different accumulators
                        const int ca = a * KS + z, cb = (k - a) * KS + z;
                        mma_ss(tmem + kLevT + (uint32_t)(k * QU),
                                   sdesc(a0 + (uint32_t)((ca >> 2) * 128 * 128 + (ca & 3) * 32)),
                                   sdesc(b0 + (uint32_t)((cb >> 2) * QU * 128 + (cb & 3) * 32)),
                                   fx_idesc(QU), (a | z) ? 1u : 0u, el);
                    }
            mma_commit(tfull, el);
            return true;
        };
        // bytes of unit u (A, in TMEM) against the V bytes of its 32 columns
        auto byte_mmas = [&](int u) -> bool {
            const int s = (u / QUG) % QNST;
            if (!mbar_wait_warp(bfull, (uint32_t)u & 1u, deadline)) return false;
            fence_after();
            const uint32_t vb = su32(sStage + (size_t)s * S::kStage + QUG * S::kB);
#pragma unroll
            for (int kk = 0; kk < QU / 16; ++kk)
#pragma unroll
                for (int a = 0; a < QNK; ++a)
                    mma_ts(tmem + kSumT, tmem + kByteT + (uint32_t)(a * (QU / 2) + kk * 8),
                               sdesc(vb + (uint32_t)((QNK - 1 - a) * CPAD * 128 +
                                                     (u % QUG) * QU * 2 + kk * 32)),
                               fx_idesc(8 * CPAD), ((u % QUG) | kk | a) ? 1u : 0u, el);
            mma_commit(bfree, el);
            if (u % QUG == QUG - 1) mma_commit(&empty[s], el);
            return true;
        };
        for (int t = 0; t < nunits && !fail; ++t)
            if (!level_mmas(t) || (t >= 1 && !byte_mmas(t - 1))) fail = 1;
        if (!fail && nunits >= 1 && !byte_mmas(nunits - 1)) fail = 1;
        mma_commit(done, el);
        if (!mbar_wait_warp(done, 0, gtimer() + kWaitNs)) fail = 1;
    } else {
        const uint32_t lane_base = tmem + ((uint32_t)(quarter * 32) << 16);
        // the byte sums of a finished group into the 32-bit sums
        auto drain = [&]() {
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const uint32_t ta = lane_base + kSumT + (uint32_t)((2 * cg + h) * CPAD);
                if constexpr (CU == 2) {
                    uint32_t r[2];
                    tmem_ld2(ta, r);
                    acc[h][0] += __float2int_rn(__uint_as_float(r[0]) * 0x1p24f);
                    acc[h][1] += __float2int_rn(__uint_as_float(r[1]) * 0x1p24f);
                } else {
#pragma unroll
                    for (int c0 = 0; c0 < CU; c0 += 8) {
                        uint32_t r[8];
                        tmem_ld4_nw(ta + c0, r);
                        tmem_ld4_nw(ta + c0 + 4, r + 4);
                        tmem_wait_ld();
                        tmem_bind4(r);
                        tmem_bind4(r + 4);
#pragma unroll
                        for (int q = 0; q < 8; ++q)
                            acc[h][c0 + q] += __float2int_rn(__uint_as_float(r[q]) * 0x1p24f);
                    }
                }
            }
        };
        constexpr int CH = CU <= 16 ? 8 : 4;  // columns loaded at a time (registers)
        // the unit whose 32 columns are this warp's 32 rows (if in this item)
        const int64_t td = rt * (128 / QU) + quarter - g0 * QUG;
        const int tdiag = td >= 0 && td < nunits ? (int)td : -1;
        for (int t = 0; t < nunits; ++t) {
            if (!__all_sync(0xffffffffu, mbar_wait(tfull, (uint32_t)t & 1u, deadline))) {
                fail = 1;
                break;
            }
            fence_after();
#pragma unroll
            for (int c0 = 0; c0 < 8; c0 += CH) {
                uint32_t r[QNS][CH];
#pragma unroll
                for (int k = 0; k < QNS; ++k)
#pragma unroll
                    for (int q = 0; q < CH; q += 4)
                        tmem_ld4_nw(lane_base + kLevT + (uint32_t)(k * QU + cg * 8 + c0 + q), &r[k][q]);
                tmem_wait_ld();
#pragma unroll
                for (int k = 0; k < QNS; ++k)
#pragma unroll
                    for (int q = 0; q < CH; q += 4) tmem_bind4(&r[k][q]);
                if (c0 + CH == 8) {  // the levels go back to the MMA thread
                    fence_before();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(tempty);
                }
#pragma unroll
                for (int q0 = 0; q0 < CH; q0 += 4) {
                    uint32_t hi[4], lo[4];
#pragma unroll
                    for (int q = 0; q < 4; ++q) {
                        const uint64_t M = fx_entry(
                            __uint_as_float(r[0][q0 + q]), __uint_as_float(r[1][q0 + q]),
                            __uint_as_float(r[2][q0 + q]), __uint_as_float(r[3][q0 + q]),
                            __uint_as_float(r[4][q0 + q]), __uint_as_float(r[5][q0 + q]), w, tab);
                        hi[q] = (uint32_t)(M >> 32);
                        lo[q] = (uint32_t)M;
                    }
                    if (t == tdiag) {  // the entries of points with themselves: 2^62
#pragma unroll
                        for (int q = 0; q < 4; ++q)
                            if (cg * 8 + c0 + q0 + q == lane) {
                                hi[q] = (1u << 30) + (uint32_t)(kDigitOff >> 32);
                                lo[q] = (uint32_t)kDigitOff;
                            }
                    }
                    if (c0 + q0 == 0 && t > 0) {
                        // the bytes of the previous unit are consumed; a finished group's
                        // sums are read before this unit's byte MMAs restart them
                        if (!__all_sync(0xffffffffu,
                                        mbar_wait(bfree, (uint32_t)(t - 1) & 1u, deadline))) {
                            fail = 1;
                            break;
                        }
                        fence_after();
                        if (t % QUG == 0) drain();
                    }
                    const uint32_t tb = lane_base + kByteT + (uint32_t)(cg * 4 + (c0 + q0) / 2);
                    // 16-bit lanes (byte, 0): columns 2 v and 2 v + 1 of the chunk
                    const uint32_t t0 = prmt(hi[0], hi[1], 0x7632), t1 = prmt(hi[2], hi[3], 0x7632);
                    const uint32_t h0 = prmt(hi[0], hi[1], 0x5410), h1 = prmt(hi[2], hi[3], 0x5410);
                    const uint32_t m0 = prmt(lo[0], lo[1], 0x7632), m1 = prmt(lo[2], lo[3], 0x7632);
                    const uint32_t l0 = prmt(lo[0], lo[1], 0x5410), l1 = prmt(lo[2], lo[3], 0x5410);
                    tmem_st2(tb + 0 * 16, prmt(t0, 0u, 0x4341), prmt(t1, 0u, 0x4341));
                    tmem_st2(tb + 1 * 16, t0 & 0x00ff00ffu, t1 & 0x00ff00ffu);
                    tmem_st2(tb + 2 * 16, prmt(h0, 0u, 0x4341), prmt(h1, 0u, 0x4341));
                    tmem_st2(tb + 3 * 16, h0 & 0x00ff00ffu, h1 & 0x00ff00ffu);
                    tmem_st2(tb + 4 * 16, prmt(m0, 0u, 0x4341), prmt(m1, 0u, 0x4341));
                    tmem_st2(tb + 5 * 16, m0 & 0x00ff00ffu, m1 & 0x00ff00ffu);
                    tmem_st2(tb + 6 * 16, prmt(l0, 0u, 0x4341), prmt(l1, 0u, 0x4341));
                    tmem_st2(tb + 7 * 16, l0 & 0x00ff00ffu, l1 & 0x00ff00ffu);
                }
                if (fail) break;
            }
            if (fail) break;
            asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
            fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(bfull);
        }
        if (!fail && nunits > 0) {
            if (!__all_sync(0xffffffffu,
                            mbar_wait(bfree, (uint32_t)(nunits - 1) & 1u, deadline))) {
                fail = 1;
            } else {
                fence_after();
                drain();
            }
        }
    }
    if (fail) atomicExch(&s_fail, 1);
    fence_before();
    __syncthreads();
    fence_after();
    // sums of levels 2 cg, 2 cg + 1 (weight 2^(-13 - 8 l)), less what the bytes' 128s have
    // put into them, smallest first, in FP64
#pragma unroll 1
    for (int g = 3; g >= 0; --g) {
        if (warp >= 2 && cg == g) {
            const double sc = ldexp(1.0, -13 - 16 * g);
#pragma unroll
            for (int k = 0; k < CU; ++k) {
                const int d0 = acc[0][k] - off[2 * g * CPAD + k];
                const int d1 = acc[1][k] - off[(2 * g + 1) * CPAD + k];
                const double v = fma((double)d1, 0x1p-8, (double)d0) * sc;
                comb[k * 128 + row] = (g == 3) ? v : comb[k * 128 + row] + v;
            }
        }
        __syncthreads();
    }
    for (int e = threadIdx.x; e < ncols * 128; e += blockDim.x)
        part[((size_t)blockIdx.y * ncols + (e >> 7)) * n_pad + rt * 128 + (e & 127)] = comb[e];
    if (threadIdx.x == 0 && s_fail) atomicExch(err, 1);
    if (warp == 1) {
        __syncwarp();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512));
    }
}

// max |x| of an array (as the bits of a non-negative double, which order as
// unsigned integers; NaN orders above infinity) and the number of its values that are
// not zero, per column k of the grid.
__global__ void fx_absmax_kernel(const double* __restrict__ x, int64_t ldx, int64_t cnt,
                                 unsigned long long* __restrict__ out,
                                 unsigned long long* __restrict__ nnz) {
    const int k = blockIdx.y;
    unsigned long long m = 0;
    unsigned c = 0;
    for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < cnt;
         e += (int64_t)gridDim.x * blockDim.x) {
        const unsigned long long b =
            (unsigned long long)__double_as_longlong(x[e + (int64_t)k * ldx]) & 0x7fffffffffffffffull;
        m = b > m ? b : m;
        c += b != 0;
    }
    c = __reduce_add_sync(0xffffffffu, c);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const unsigned long long q = __shfl_xor_sync(0xffffffffu, m, o);
        m = q > m ? q : m;
    }
    if ((threadIdx.x & 31) == 0 && m) {
        atomicMax(&out[k], m);
        atomicAdd(&nnz[k], (unsigned long long)c);
    }
}

// Byte offset of element (r, k) inside a rows x 64 swizzled K-major sub-tile.
__device__ __forceinline__ uint32_t fx_swz(int r, int k) {
    return (uint32_t)(r * 128 + (((k >> 3) ^ (r & 7)) * 16) + (k & 7) * 2);
}

// One thread per point: its row of A (tiles of 128 rows) and of B (units of 32).
// scale_h + scale_l = sqrt(log2 e) in two doubles; the slices are cut from the
// unrounded product xs64 * sqrt(log2 e) / S.
template <int KS>
__global__ void fx_prep_kernel(const double* __restrict__ xs64, int64_t n, int64_t n_pad, int dp,
                               int d, double scale_h, double scale_l, double invS9,
                               uint8_t* __restrict__ Aop, uint8_t* __restrict__ Bop) {
    constexpr int SUBT = (QNS * KS + 3) / 4;
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n_pad) return;
    uint8_t* ab = Aop + (size_t)(i / 128) * SUBT * 128 * 128;
    uint8_t* bb = Bop + (size_t)(i / QU) * SUBT * QU * 128;
    const int ar = (int)(i % 128), br = (int)(i % QU);
    auto put = [&](int a, int k, float va, float vb) {
        const int c = a * KS * 16 + k;
        *reinterpret_cast<__half*>(ab + (size_t)(c >> 6) * 128 * 128 + fx_swz(ar, c & 63)) =
            __float2half_rn(va);
        *reinterpret_cast<__half*>(bb + (size_t)(c >> 6) * QU * 128 + fx_swz(br, c & 63)) =
            __float2half_rn(vb);
    };
    int s[QNS][16];
    for (int r = 0; r < 16; ++r) {
        double h = 0.0, l = 0.0;
        if (i < n && r < d) {
            const double x = xs64[i * dp + r];
            const double p = x * scale_h;
            l = (fma(x, scale_h, -p) + x * scale_l) * invS9;
            h = p * invS9;
        }
        for (int a = 0; a < QNS; ++a) {
            const double v = rint(h);
            s[a][r] = (int)v;
            h -= v;
            if (a == 0) h += l;
            h *= 1024.0;
        }
    }
    // N = |y|^2 over all levels, in units of the last one kept; ceil(N / 2) as
    // balanced base-1024 digits (the top one as 1024 h + l)
    __int128 N = 0;
    double rest = 0.0;
    for (int k = 0; k < 2 * QNS - 1; ++k) {
        long long L = 0;
        for (int a = max(0, k - QNS + 1); a <= min(k, QNS - 1); ++a)
            for (int r = 0; r < d; ++r) L += (long long)s[a][r] * s[k - a][r];
        if (k < QNS)
            N = N * 1024 + L;
        else
            rest += (double)L * ldexp(1.0, -10 * (k - QNS + 1));
    }
    N = (N + (long long)rint(rest) + 1) >> 1;
    int nd[QNS];
    for (int k = QNS - 1; k >= 1; --k) {
        const int v = (int)((long long)((N + 512) & 1023)) - 512;
        nd[k] = -v;
        N = (N - v) >> 10;
    }
    const int n0 = (int)N;
    const int hN = (n0 + 512) >> 10;
    nd[0] = -(n0 - hN * 1024);
    for (int a = 0; a < QNS; ++a) {
        for (int r = 0; r < KS * 16; ++r) {
            float va = 0.f, vb = 0.f;
            if (i < n) {
                if (r < d)
                    va = vb = (float)s[a][r];
                else if (r == d) {
                    va = a == 0 ? 1.f : 0.f;
                    vb = (float)nd[a];
                } else if (r == d + 1) {
                    va = a == 0 ? 1024.f : 0.f;
                    vb = a == 0 ? (float)-hN : 0.f;
                } else if (r == d + 2) {
                    va = (float)nd[a];
                    vb = a == 0 ? 1.f : 0.f;
                } else if (r == d + 3) {
                    va = a == 0 ? (float)-hN : 0.f;
                    vb = a == 0 ? 1024.f : 0.f;
                }
            }
            put(a, r, va, vb);
        }
    }
    for (int c = QNS * KS * 16; c < SUBT * 64; ++c) put(c / (KS * 16), c % (KS * 16), 0.f, 0.f);
}

// V's columns as eight balanced bytes each, v = 2^e sum_b v_b 2^(-7 - 8b), 2^e > max|v|:
// per group of 64 rows of V, operand rows (b, column) of 64 FP16, swizzled.  One
// thread per (group, column, 8 rows).  vsum[group][l][column] = 128 sum of the bytes b < l over
// the group.  Columns with few values or one that is not finite are left zero (the
// reduction computes them entry by entry); the few values go to their list.
__global__ void fx_stage_v_kernel(const double* __restrict__ V, int64_t ldv, int64_t n,
                                  int64_t n_pad, int ncols, int cpad,
                                  FxCols* __restrict__ cols, uint8_t* __restrict__ Vop,
                                  int* __restrict__ vsum) {
    const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= (n_pad / 8) * cpad) return;
    // consecutive threads: the 8-row chunks of a column (coalesced reads)
    const int64_t chunk = e % (n_pad / 8);
    const int k = (int)(e / (n_pad / 8));
    const int64_t g = chunk >> 3;
    const int c8 = (int)(chunk & 7);
    uint32_t out[QNV][4];
    float sum[QNV];  // at most 64 x 128 over a group
#pragma unroll
    for (int b = 0; b < QNV; ++b) {
        sum[b] = 0.f;
#pragma unroll
        for (int w = 0; w < 4; ++w) out[b][w] = 0u;
    }
    const bool few = k < ncols && cols->nnz[k] <= kFew;
    if (few) {
#pragma unroll 1
        for (int64_t j = chunk * 8; j < min(n, chunk * 8 + 8); ++j) {
            const double v = V[j + (int64_t)k * ldv];
            if (v != 0.0) {
                const unsigned at = atomicAdd(&cols->got[k], 1u);
                if (at < kFew) {
                    cols->row[k][at] = (int)j;
                    cols->val[k][at] = v;
                }
            }
        }
    } else if (k < ncols && cols->mx[k] < 0x7ff0000000000000ull) {
        int ex;
        (void)frexp(__longlong_as_double((long long)cols->mx[k]), &ex);
#pragma unroll
        for (int r = 0; r < 8; ++r) {
            const int64_t j = chunk * 8 + r;
            double h = j < n ? ldexp(V[j + (int64_t)k * ldv], 7 - ex) : 0.0;
#pragma unroll
            for (int b = 0; b < QNV; ++b) {
                const double v = rint(h);
                h = (h - v) * 256.0;
                const float vf = (float)v;
                sum[b] += vf;
                const uint32_t bits = __half_as_ushort(__float2half_rn(vf));
                out[b][r >> 1] |= bits << (16 * (r & 1));
            }
        }
    }
#pragma unroll
    for (int b = 0; b < QNV; ++b) {
        const int rr = b * cpad + k;
        *reinterpret_cast<uint4*>(Vop + ((size_t)g * QNV * cpad + rr) * 128 + ((c8 ^ (rr & 7)) * 16)) =
            make_uint4(out[b][0], out[b][1], out[b][2], out[b][3]);
    }
    // over the group's eight threads, neighbours of a warp (n_pad / 8 is a multiple of 16)
    int above = 0;
#pragma unroll
    for (int b = 0; b < QNV; ++b) {
#pragma unroll
        for (int o = 4; o > 0; o >>= 1) sum[b] += __shfl_xor_sync(0xffffffffu, sum[b], o);
        if (c8 == 0) vsum[((size_t)g * QNV + b) * cpad + k] = 128 * above;
        above += (int)sum[b];
    }
}

// K_ij in FP64
__device__ __forceinline__ double fx_entry64(const double* __restrict__ xs64, int dp, double c0,
                                             int64_t i, int64_t j) {
    double a = c0;
    for (int r = 0; r < dp; ++r) {
        const double t = xs64[i * dp + r] - xs64[j * dp + r];
        a = fma(-t, t, a);
    }
    return exp(fmax(a, -708.0));
}

// O = s^2 2^e (sum of the split partials) + noise V, or B minus that, in FP64.  A column of at
// most kFew values (a unit vector asks for a column of K, whose entries a cut at an absolute
// place would not give) is a sum of FP64 entries in the order of the rows: 0.1 ms of FP64 at
// n = 65536 with all 32.
__global__ void fx_reduce_kernel(const double* __restrict__ part, int64_t n_pad, int nsplit,
                                 int ncols, const FxCols* __restrict__ cols, double s2,
                                 const double* __restrict__ xs64, int dp, double c0,
                                 const double* __restrict__ V, int64_t ldv, double noise,
                                 const double* __restrict__ B, int64_t ldb, double* __restrict__ O,
                                 int64_t ldo, int64_t n) {
    __shared__ int rows[kFew];
    __shared__ double vals[kFew];
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int k = blockIdx.y;
    const unsigned long long mx = cols->mx[k], nnz = cols->nnz[k];
    const int nf = nnz <= kFew ? (int)nnz : -1;
    if (nf >= 0) {  // its values in the order of the rows
        if ((int)threadIdx.x < nf) {
            const int row = cols->row[k][threadIdx.x];
            int rank = 0;
            for (int u = 0; u < nf; ++u) rank += cols->row[k][u] < row;
            rows[rank] = row;
            vals[rank] = cols->val[k][threadIdx.x];
        }
        __syncthreads();
    }
    if (i >= n) return;
    double s = 0.0;
    if (nf >= 0) {
        for (int u = 0; u < nf; ++u) s = fma(fx_entry64(xs64, dp, c0, i, rows[u]), vals[u], s);
    } else if (mx < 0x7ff0000000000000ull) {
        for (int sp = 0; sp < nsplit; ++sp) s += part[((size_t)sp * ncols + k) * n_pad + i];
        // one power of two for V and s^2: neither alone may leave the range that O keeps
        int ex = 0, e2 = 0;
        (void)frexp(__longlong_as_double((long long)mx), &ex);
        s = ldexp(frexp(s2, &e2) * s, ex + e2);
    } else {
        // an infinity or a NaN in the column: every entry in FP64, as IEEE has it
        for (int64_t j = 0; j < n; ++j)
            s = fma(fx_entry64(xs64, dp, c0, i, j), V[j + (int64_t)k * ldv], s);
    }
    s = fma(noise, V[i + (int64_t)k * ldv], s);
    O[i + (int64_t)k * ldo] = B ? (B[i + (int64_t)k * ldb] - s) : s;
}

template <int SUBT, int KS, int CPAD, int CU>
void launch_fx(Ctx& h, const uint8_t* Vop, const int* vsum, int64_t n_pad, int ncols, int nsplit, int gps,
               double* part, uint64_t wait_ns) {
    using S = FxSmem<SUBT, CPAD>;
    allow_smem(kv_fx_kernel<SUBT, KS, CPAD, CU>, S::kTotal);
    const float w0 = (float)std::ldexp(h.fx_S * h.fx_S, -17);
    const FxScale w{w0, w0 * 0x1p-10f, w0 * 0x1p-20f, w0 * 0x1p-30f, w0 * 0x1p-40f};
    kv_fx_kernel<SUBT, KS, CPAD, CU><<<dim3((unsigned)(n_pad / 128), (unsigned)nsplit), QWARPS * 32,
                                   S::kTotal, h.stream>>>(
        reinterpret_cast<const __half*>(h.fxA.p), reinterpret_cast<const __half*>(h.fxB.p),
        reinterpret_cast<const __half*>(Vop), vsum, h.n, n_pad, ncols, gps, w, h.fx_tab.p, part,
        h.tc_err.p, wait_ns, h.opt.wait_stall ? 1 : 0);
    KPCG_LAUNCHED("kv_fx_kernel");
}

template <int CPAD, int CU>
void launch_fx_ks(Ctx& h, const uint8_t* Vop, const int* vsum, int64_t n_pad, int ncols, int nsplit, int gps,
                  double* part, uint64_t wait_ns) {
    if (h.d + 4 <= 16)
        launch_fx<2, 1, CPAD, CU>(h, Vop, vsum, n_pad, ncols, nsplit, gps, part, wait_ns);
    else
        launch_fx<3, 2, CPAD, CU>(h, Vop, vsum, n_pad, ncols, nsplit, gps, part, wait_ns);
}

// floor(sqrt(v))
uint64_t isqrt128(unsigned __int128 v) {
    uint64_t r = 0;
    for (int b = 63; b >= 0; --b) {
        const uint64_t t = r | ((uint64_t)1 << b);
        if ((unsigned __int128)t * t <= v) r = t;
    }
    return r;
}

// round(2^(56 - j/4096)) - kTabOff, j = 0 .. 4095, in integers: 2^(-2^b/4096) by
// repeated square roots with 64 fraction bits, their products over the bits of j.
std::vector<uint64_t> fx_table() {
    uint64_t root[12];
    root[11] = isqrt128((unsigned __int128)1 << 127);
    for (int b = 10; b >= 0; --b) root[b] = isqrt128((unsigned __int128)root[b + 1] << 64);
    std::vector<uint64_t> t(QTAB);
    for (int j = 0; j < QTAB; ++j) {
        unsigned __int128 v = (unsigned __int128)1 << 64;
        for (int b = 0; b < 12; ++b)
            if (j >> b & 1) v = (v * root[b] + ((unsigned __int128)1 << 63)) >> 64;
        t[(size_t)j] = (uint64_t)((v + 128) >> 8) - kTabOff;
    }
    return t;
}

// The scale S of the handle's current theta: the power of two from max |y| up.
void fx_prepare(Ctx& h) {
    if (h.fx_version == h.theta_version) return;
    cudaStream_t st = h.stream;
    const int64_t n = h.n;
    FxCols* cols = reinterpret_cast<FxCols*>(h.fxCols.need(sizeof(FxCols)));
    unsigned long long* mx = cols->mx;
    KPCG_CUDA(cudaMemsetAsync(mx, 0, sizeof(unsigned long long), st));
    const int64_t cnt = n * h.dp;
    fx_absmax_kernel<<<(unsigned)std::min<int64_t>((cnt + 1023) / 1024, 608), 256, 0, st>>>(
        h.xs64.p, 0, cnt, mx, cols->nnz);
    KPCG_LAUNCHED("fx_absmax_kernel");
    unsigned long long bits = 0;
    KPCG_CUDA(cudaMemcpyAsync(&bits, mx, sizeof(bits), cudaMemcpyDeviceToHost, st));
    KPCG_CUDA(cudaStreamSynchronize(st));
    double xmax;
    static_assert(sizeof(xmax) == sizeof(bits), "");
    std::memcpy(&xmax, &bits, sizeof(xmax));
    xmax *= std::sqrt(kLog2e) * (1.0 + 1e-15);
    // at least 2: below that the leading levels of r no longer fit 24 bits
    double S = 2.0;
    while (S < xmax && S < 0x1p40) S *= 2.0;
    h.fx_S = (std::isfinite(xmax) && S < 0x1p40) ? S : INFINITY;
    h.fx_version = h.theta_version;
    h.fx_op_version = -1;
}

// Operands for the scale found by fx_prepare.
void fx_operands(Ctx& h, int64_t n_pad) {
    if (h.fx_op_version == h.theta_version) return;
    cudaStream_t st = h.stream;
    if (!h.fx_tab.p) {
        const std::vector<uint64_t> t = fx_table();
        uint64_t* p = h.fx_tab.need(QTAB);
        KPCG_CUDA(cudaMemcpyAsync(p, t.data(), sizeof(uint64_t) * QTAB, cudaMemcpyHostToDevice, st));
        KPCG_CUDA(cudaStreamSynchronize(st));  // the host table leaves scope
    }
    if (!h.tc_err.p) {
        int* e = h.tc_err.need(1);
        KPCG_CUDA(cudaMemsetAsync(e, 0, sizeof(int), st));
    }
    const bool one = h.d + 4 <= 16;
    const size_t bytes = (size_t)n_pad * (one ? 2 : 3) * 128;
    uint8_t* A = h.fxA.need(bytes);
    uint8_t* Bm = h.fxB.need(bytes);
    // sqrt(log2 e) in two doubles
    constexpr double kSh = 0x1.337cc2183b050p+0, kSl = -0x1.10e9cb301c4a4p-55;
    const double invS9 = 512.0 / h.fx_S;
    const unsigned grid = (unsigned)((n_pad + 127) / 128);
    if (one)
        fx_prep_kernel<1><<<grid, 128, 0, st>>>(h.xs64.p, h.n, n_pad, h.dp, h.d, kSh, kSl, invS9, A, Bm);
    else
        fx_prep_kernel<2><<<grid, 128, 0, st>>>(h.xs64.p, h.n, n_pad, h.dp, h.d, kSh, kSl, invS9, A, Bm);
    KPCG_LAUNCHED("fx_prep_kernel");
    h.fx_op_version = h.theta_version;
}

// Splits of the column range: the split whose whole waves of work items (one per
// SM) take least, an item costing its groups plus about three more for its start
// (table and A tile into shared memory) and end.
void fx_split(int64_t n_pad, int& nsplit, int& gps) {
    const int64_t rows = n_pad / 128, groups = n_pad / QG;
    const int sms = sm_count_tc();
    double best = 1e300;
    nsplit = 1;
    for (int64_t ns = (groups + kMaxGroups - 1) / kMaxGroups, e = 0; ns <= groups && e < 64; ++ns, ++e) {
        const int64_t per = (groups + ns - 1) / ns;
        const int64_t got = (groups + per - 1) / per;
        const double cost = std::ceil((double)(rows * got) / sms) * (double)(per + 3);
        if (cost < best * 0.999) {
            best = cost;
            nsplit = (int)got;
        }
    }
    gps = (int)((groups + nsplit - 1) / nsplit);
    nsplit = (int)((groups + gps - 1) / gps);
}

// columns per pass of a block of c, in passes of nearly equal width
int fx_pass(int c) {
    const int np = (c + QMAXC - 1) / QMAXC;
    return (c + np - 1) / np;
}

}  // namespace

// Whether kv_fx serves the handle: d <= 16, the scale S at most smax (the dropped
// levels cost ~2^-59 S^2 of an exponent), partial sums within 4 GiB.
bool kv_fx_usable(Ctx& h, int c, double smax) {
    if (h.d < 1 || h.d > 16 || h.n < 1) return false;
    const int64_t n_pad = (h.n + 127) / 128 * 128;
    int nsplit, gps;
    fx_split(n_pad, nsplit, gps);
    if ((double)nsplit * fx_pass(c) * (double)n_pad * 8.0 > 4.0 * 1024 * 1024 * 1024) return false;
    fx_prepare(h);
    return h.fx_S <= smax;
}

void kv_fx(Ctx& h, const double* V, int64_t ldv, int c, const double* B, int64_t ldb, double* O,
           int64_t ldo, double noise, bool limited) {
    if (h.n <= 0 || c <= 0) return;
    cudaStream_t st = h.stream;
    const int64_t n = h.n, n_pad = (n + 127) / 128 * 128;
    const uint64_t wait_ns = (limited || h.opt.wait_stall) && h.opt.wait_limit_ns > 0
                                 ? (uint64_t)h.opt.wait_limit_ns
                                 : kWaitNs;
    fx_prepare(h);
    fx_operands(h, n_pad);
    int nsplit, gps;
    fx_split(n_pad, nsplit, gps);
    const int step = fx_pass(c);
    const int cpad = step <= 8 ? 8 : step <= 16 ? 16 : 24;
    uint8_t* Vop = h.fxV.need((size_t)(n_pad / QG) * QNV * cpad * 128);
    int* vsum = h.fxVsum.need((size_t)(n_pad / QG) * QNV * cpad);
    double* part = h.fxPart.need((size_t)nsplit * step * n_pad);
    FxCols* cols = reinterpret_cast<FxCols*>(h.fxCols.need(sizeof(FxCols)));
    for (int k0 = 0; k0 < c; k0 += step) {
        const int nc = std::min(step, c - k0);
        const double* Vk = V + (int64_t)k0 * ldv;
        KPCG_CUDA(cudaMemsetAsync(cols, 0, offsetof(FxCols, row), st));
        fx_absmax_kernel<<<dim3((unsigned)std::min<int64_t>((n + 1023) / 1024, 152), (unsigned)nc),
                           256, 0, st>>>(Vk, ldv, n, cols->mx, cols->nnz);
        KPCG_LAUNCHED("fx_absmax_kernel");
        const int64_t thr = (n_pad / 8) * cpad;
        fx_stage_v_kernel<<<(unsigned)((thr + 127) / 128), 128, 0, st>>>(Vk, ldv, n, n_pad, nc, cpad,
                                                                         cols, Vop, vsum);
        KPCG_LAUNCHED("fx_stage_v_kernel");
        // V is staged at the call's width: a narrow last pass of a wide block keeps that layout
        if (cpad == 8 && nc <= 2)
            launch_fx_ks<8, 2>(h, Vop, vsum, n_pad, nc, nsplit, gps, part, wait_ns);
        else if (cpad == 8)
            launch_fx_ks<8, 8>(h, Vop, vsum, n_pad, nc, nsplit, gps, part, wait_ns);
        else if (cpad == 16)
            launch_fx_ks<16, 16>(h, Vop, vsum, n_pad, nc, nsplit, gps, part, wait_ns);
        else
            launch_fx_ks<24, 24>(h, Vop, vsum, n_pad, nc, nsplit, gps, part, wait_ns);
        fx_reduce_kernel<<<dim3((unsigned)((n + 127) / 128), (unsigned)nc), 128, 0, st>>>(
            part, n_pad, nsplit, nc, cols, h.s2, h.xs64.p, h.dp, h.c0_64(), Vk, ldv, noise,
            B ? B + (int64_t)k0 * ldb : nullptr, ldb, O + (int64_t)k0 * ldo, ldo, n);
        KPCG_LAUNCHED("fx_reduce_kernel");
    }
}

}  // namespace kpcg

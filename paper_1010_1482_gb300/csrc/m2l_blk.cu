// M2L (Eq. 4) of the uniform tree as a block convolution on the tcgen05 tensor cores.
//
// On the uniform tree the M2L list of a level-l cell t = 2Q + tau (Q its parent's integer
// coordinates, tau its child position) holds the children sigma of the parent's 26 neighbours
// S = Q + D whose offset o = 2D + sigma - tau is not a near neighbour (|o|_inf >= 2).  Grouped by
// the parent offset D, the M2L of all 8 children of Q is
//     L~(Q, tau) = sum_D sum_sigma B_D[tau][sigma] M~(Q + D, sigma),
//     B_D[tau][sigma] = T_{2D + sigma - tau} if |2D + sigma - tau|_inf >= 2, else 0,
// where T_o is the p^2 x p^2 real M2L operator of offset o (Eq. 4-6, scaled expansions).  Over
// the parents of a level this is one dense GEMM per D:
//     D[Q][(tau, n)] += sum_(sigma, k) A[Q + D][(sigma, k)] B_D[(tau, n)][(sigma, k)],
// A[S] = the 8 p^2 multipole coefficients of the children of parent S (zero for empty cells and
// for S outside the level).  K = N = 8 p^2 (800 at p = 10): no padding, and the zero blocks of
// B_D (near pairs) are 9% of its entries.  No interaction lists are read.
//
// Parity classes.  Mirroring an axis maps child sigma to its mirror image and multiplies every
// real-packed coefficient by a sign s(n, m, re/im) (T_{R o} = S_R T_o S_R), so with the children's
// coefficients combined into sums and differences over each axis,
//     U_c[k] = sum_sigma (-1)^{c . sigma} s(k)^sigma M~_sigma[k],   c in {0, 1}^3,
// class c has a definite parity in every axis, and B'_D = H B_D H^T / 8 couples class c' of the
// targets with class c of the sources only where they agree in every axis along which D is 0.  H is
// orthogonal up to the factor 8, so nothing is lost: L~ = H^T V / 8.  A CTA's N-tile is one unit of
// classes (all of them agree in the axes that distinguish units), and per D it walks only the
// units of K that its own couples with: at p = 10 (units of two classes) 148 of 208 class products
// over the 26 offsets, at p = 6 and 8 (four classes) 176.  The pre-split kernels form U, the drains
// write V, and a last kernel (k_blk_finish, k_ablk_finish) adds the offset ranges and applies H^T.
// Against the untransformed blocks: M2L kernel of 1M uniform, p = 10 321 -> 266 us (the step 1022 ->
// 969), of 400,009 Plummer, p = 10 549 -> 398; 16M Plummer, p = 8 step 23.21 -> 22.56 ms, a batch of
// 96 instances 7.05 -> 6.62 ms.  Bound by shared memory: a K step of 16 at p = 10 reads 31 KB of
// operands and takes 21 KB of copies in 312 cycles of MMA, 167 bytes a cycle of 128.
//
// Tiles: one CTA takes 128 target parents (a box of 8 x 4 x 4 in the parent grid; smaller on
// levels 2 and 3) as the MMA's M and one N-tile of the 8 p^2 outputs, and walks the 26 offsets
// D in chunks of 32 or 64 K values.  Operands stream through shared memory by TMA tiled loads
// (the source box shifted by D, out-of-range parents zero-filled; B_D's N-tile), swizzled,
// and both are read by the MMA from shared memory.  Precision is the 3xF16 scheme of the
// gathered kernel: x = hi + lo in FP16, D += A_lo B_hi + A_hi B_lo + A_hi B_hi with FP32
// accumulation in TMEM.  Scales: every source parent's coefficients by 2^s_S (max -> 2^10), the
// operators by one power of two 2^g (max over all offsets -> 2^12).  Each D's partial is drained
// from TMEM (DPU pieces a unit, bounding the truncating accumulation chain) to FP32 registers
// and multiplied by 2^-(s_(Q+D) + g) per row before the sum; two TMEM accumulators alternate so
// the MMAs of the next piece overlap the drain.
#include "common.cuh"
#include "ptx.cuh"

#include <cuda.h>
#include <cuda_fp16.h>
#include <cudaTypedefs.h>

#include <cstring>
#include <mutex>

namespace gbfmm {

namespace {

constexpr int kBlkRows = 128;  // target parents per CTA (MMA M)
constexpr int kBlkDrainWarps = 8;
constexpr int kBlkThreads = 32 * (kBlkDrainWarps + 2);  // drain warps, TMA producer, MMA issuer

// the 26 parent offsets D in {-1, 0, 1}^3 \ {0}: index d -> D
GB_HD void blk_delta(int d, int &dx, int &dy, int &dz)
{
    const int i = d < 13 ? d : d + 1;
    dx = i % 3 - 1;
    dy = (i / 3) % 3 - 1;
    dz = i / 9 - 1;
}

}  // namespace

// K values per pipeline stage, one shared-memory row of 64 bytes (64-byte swizzle).  Four stages of 32
// cover the copies' latency better at p = 10 than two of 64 (M2L of 1M, 343 us against 372 before the
// parity classes).  At p = 4 and 6 three stages of 64 run the M2L alone faster (5M: 174 us against 135
// and 534 against 438; 400,009 Plummer 97 against 93 and 165 against 159), but take the room of a P2P
// CTA beside them: the step gains little or loses (p = 4 1M 613 : 612, 5M 2310 : 2285; p = 6 1M 661 :
// 670, 5M 2685 : 2689, 400,009 Plummer 790 : 785), and at p = 4 a chunk of 64 doubles the longest
// accumulation chain, and with it the error (see DPU).
constexpr int kBlkCh = 32;

template <int P>
struct BlkCfg {
    static constexpr int PP = P * P, KD = 8 * PP;
    // N-tile: rows of B_D per CTA (the MMA's N, a multiple of 16) and the stride between tiles
    static constexpr int NT = P == 4 ? 128 : P == 6 ? 144 : P == 8 ? 256 : 208;
    // units of classes: CU classes, UNIT K values (padded to the MMA's 16); K rows hold the units in
    // order (class c, coefficient k at (c / CU) UNIT + (c % CU) PP + k), an N-tile is one unit
    static constexpr int CU = P == 10 ? 2 : P == 4 ? 8 : 4, NUNIT = 8 / CU;
    static constexpr int UNIT = (CU * PP + 15) / 16 * 16, KW = NUNIT * UNIT;
    static constexpr int NSTRIDE = CU * PP, NTILES = NUNIT;
    static constexpr int UC = (UNIT + kBlkCh - 1) / kBlkCh;  // chunks of a unit
    // drains per unit: the MMA's accumulation truncates, and a class sums eight children.  Chains of
    // 6, 18, 24 and 39 MMAs at p = 4, 6, 8, 10 leave the outputs as close to the FP64 FMM as, or
    // closer than, the untransformed blocks with chains of 12, 27, 48 and 75 did (phi, 30,000 uniform
    // particles: 1.7, 3.5, 3.5, 3.7e-7 against 1.9, 3.7, 4.3, 5.3e-7); twice as long at p = 4: 2.4e-7
    static constexpr int DPU = P == 10 ? 1 : P == 4 ? 4 : 2;
    static constexpr int MAX_STEPS = 26 * NUNIT * UC, MAX_DRAINS = 26 * NUNIT * DPU;
    static constexpr int A_BYTES = kBlkRows * kBlkCh * 2;  // one of hi / lo
    static constexpr int B_BYTES = NT * kBlkCh * 2;
    static constexpr int STAGE_BYTES = 2 * A_BYTES + 2 * B_BYTES;
    static constexpr int NSTAGE_FIT = (210 * 1024) / STAGE_BYTES;
    static constexpr int NSTAGE = NSTAGE_FIT > 4 ? 4 : NSTAGE_FIT;
    static constexpr size_t kSmemBytes = (size_t)NSTAGE * STAGE_BYTES + 1024;  // + alignment slack
    static constexpr int NH = NT / 2;  // accumulator columns per drain thread
    static constexpr int TMEM_COLS = 2 * NT <= 256 ? 256 : 512;
    static_assert(NT % 16 == 0 && NT <= 256, "MMA N");
    static_assert(NH % 8 == 0 && NSTRIDE % 4 == 0 && PP % 4 == 0, "drain / store granularity");
    static_assert(NSTRIDE <= NT && NTILES * NSTRIDE == KD, "N tiling");
    static_assert(UNIT % 16 == 0 && KW % 8 == 0 && UC >= DPU && MAX_DRAINS < 1024, "steps");
    static_assert(A_BYTES % 1024 == 0 && B_BYTES % 1024 == 0, "swizzle atoms");
    static_assert(2 * kBlkCh == 64, "the row of the 64-byte swizzle (descriptors, tensor maps, loaders)");
    static_assert(NSTAGE >= 2, "pipeline stages");
    static_assert(kSmemBytes <= 227 * 1024, "shared memory");
};

// the axes' signs of coefficient k (real-packed, degree n at n^2: m = 0, then re, im of m = 1, 2, ...)
// under a mirror in x, y, z, as a bit mask of the negative ones
GB_HD int blk_signs(int k)
{
    int n = 0;
#pragma unroll
    for (int j = 1; j < 10; ++j) n += k >= j * j;
    const int r = k - n * n, m = (r + 1) / 2, sy = (r > 0 && r % 2 == 0) ? 1 : 0;
    return ((m & 1) ^ sy) | sy << 1 | ((n + m) & 1) << 2;
}

// v[sigma] -> sum_sigma (-1)^{c . sigma} v[sigma], c = 0..7
GB_DEV void blk_hadamard(float (&v)[8])
{
#pragma unroll
    for (int b = 1; b < 8; b <<= 1)
#pragma unroll
        for (int i = 0; i < 8; ++i)
            if (!(i & b)) {
                const float x = v[i], y = v[i | b];
                v[i] = x + y;
                v[i | b] = x - y;
            }
}

// v[sigma] *= s^sigma
GB_DEV void blk_sign_children(float (&v)[8], int signs)
{
#pragma unroll
    for (int i = 0; i < 8; ++i)
        if (__popc(i & signs) & 1) v[i] = -v[i];
}

// One CTA's pipeline: per step (K chunk) the offset, first K value, width and whether it opens or
// closes a drain unit; the units' offsets.  Built by one warp before the roles part.
template <class C>
struct BlkSteps {
    uint32_t step[C::MAX_STEPS];  // d | k0 / 8 << 5 | kw / 16 << 13 | first << 16 | last << 17 | drain << 18
    uint8_t drain_d[C::MAX_DRAINS];
    int nsteps, ndrains;
};
GB_DEV int step_d(uint32_t v) { return v & 31; }
GB_DEV int step_k0(uint32_t v) { return (int)(v >> 5 & 255) * 8; }
GB_DEV int step_kw(uint32_t v) { return (int)(v >> 13 & 7) * 16; }
GB_DEV bool step_first(uint32_t v) { return v >> 16 & 1; }
GB_DEV bool step_last(uint32_t v) { return v >> 17 & 1; }
GB_DEV int step_drain(uint32_t v) { return (int)(v >> 18); }

// one warp; nt: the CTA's unit of classes, offsets [d_lo, d_hi)
template <class C>
GB_DEV void blk_steps(BlkSteps<C> &t, int nt, int d_lo, int d_hi, int lane)
{
    constexpr int UB = C::NUNIT == 4 ? 2 : C::NUNIT == 2 ? 1 : 0;  // axes that distinguish units: the last UB
    const int d = d_lo + lane;
    int dx = 0, dy = 0, dz = 0, free = 0;
    if (d < d_hi) {
        blk_delta(d, dx, dy, dz);
        free = UB == 2 ? (dy != 0) | (dz != 0) << 1 : UB == 1 ? (dz != 0) : 0;
    }
    const int nun = d < d_hi ? 1 << __popc(free) : 0;
    int su = nun;  // inclusive scan
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int a = __shfl_up_sync(~0u, su, o);
        if (lane >= o) su += a;
    }
    int i = su - nun;  // units before, of all the CTA's offsets
    for (int e = 0; e < C::NUNIT; ++e) {
        if (nun == 0 || (e & ~free)) continue;
        const int ku = nt ^ e;
        for (int c = 0; c < C::UC; ++c) {
            const int kw = min(kBlkCh, C::UNIT - c * kBlkCh), piece = c * C::DPU / C::UC, dr = i * C::DPU + piece;
            const bool first = c == 0 || (c - 1) * C::DPU / C::UC != piece;
            const bool last = c == C::UC - 1 || (c + 1) * C::DPU / C::UC != piece;
            if (first) t.drain_d[dr] = (uint8_t)d;
            t.step[i * C::UC + c] = (uint32_t)d | (uint32_t)((ku * C::UNIT + c * kBlkCh) / 8) << 5 | (uint32_t)(kw / 16) << 13 |
                                    (uint32_t)first << 16 | (uint32_t)last << 17 | (uint32_t)dr << 18;
        }
        ++i;
    }
    if (lane == 31) t.nsteps = su * C::UC, t.ndrains = su * C::DPU;
}

constexpr size_t blk_kw(int P)  // K row width
{
    return P == 4 ? BlkCfg<4>::KW : P == 6 ? BlkCfg<6>::KW : P == 8 ? BlkCfg<8>::KW
                                                                                  : BlkCfg<10>::KW;
}

// tensor maps and tiling of one launch (kernel parameter, read by the TMA unit in place)
struct BlkParams {
    CUtensorMap tmA[kMaxLevel + 1];  // per target level l: the presplit sources of the level's children
    CUtensorMap tmB;                 // B_D, FP16 hi | lo
    int L;
    int tile_lo[kMaxLevel + 2];      // tiles of level l: [tile_lo[l], tile_lo[l + 1]) (levels in ascending order)
    int tile0;                       // tile of block 0 (launch in waves)
    int ksplit;                      // the 26 offsets are split into ksplit ranges, one per CTA
    int64_t part_stride;             // ksplit > 1: floats between the partial sums of two ranges
};

// ---- shared-memory matrix descriptor, K-major, swizzled -----------------------------------------
// rows of 64 bytes, 8-row atoms of 512 bytes (SBO); a K step of 16 halves advances the start
// address by 32 bytes inside the atom.  Swizzle mode: 4 = 64-byte.
GB_DEV uint64_t blk_desc(uint32_t saddr)
{
    uint64_t d = (uint64_t)((saddr & 0x3FFFFu) >> 4);
    d |= (uint64_t)1 << 16;                     // LBO (unused for swizzled K-major operands)
    d |= (uint64_t)((16 * kBlkCh) >> 4) << 32;  // SBO: 8-row atoms
    d |= (uint64_t)1 << 46;                     // descriptor version of the 5th-generation tensor cores
    d |= (uint64_t)4 << 61;                     // swizzle mode
    return d;
}

GB_DEV void blk_mma_ss(uint32_t d_tmem, uint64_t adesc, uint64_t bdesc, uint32_t idesc, uint32_t accumulate)
{
    asm volatile(
        "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
        " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(d_tmem),
        "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate)
        : "memory");
}

GB_DEV void blk_tma5(void *dst, const CUtensorMap *tm, int c0, int c1, int c2, int c3, int c4, uint64_t *bar)
{
    asm volatile(
        "cp.async.bulk.tensor.5d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4, %5, "
        "%6}], [%7];" ::"r"(smem_u32(dst)),
        "l"(reinterpret_cast<uint64_t>(tm)), "r"(c0), "r"(c1), "r"(c2), "r"(c3), "r"(c4), "r"(smem_u32(bar))
        : "memory");
}

GB_DEV void blk_tma4(void *dst, const CUtensorMap *tm, int c0, int c1, int c2, int c3, uint64_t *bar)
{
    asm volatile(
        "cp.async.bulk.tensor.4d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4, %5}], "
        "[%6];" ::"r"(smem_u32(dst)),
        "l"(reinterpret_cast<uint64_t>(tm)), "r"(c0), "r"(c1), "r"(c2), "r"(c3), "r"(smem_u32(bar))
        : "memory");
}

GB_DEV void blk_prefetch_tmap(const CUtensorMap *tm)
{
    asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(tm)) : "memory");
}

// whole warp: 8 consecutive 32-bit columns of the thread's TMEM lane, no wait
GB_DEV void blk_ld8(uint32_t taddr, uint32_t *v)
{
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
                 : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7])
                 : "r"(taddr));
}

// 2^e as a float (e within the normal range)
GB_DEV float blk_pow2(int e) { return __int_as_float((127 + e) << 23); }

// ---- pre-split sources: per parent S of levels 1 .. L - 1, in grid order (x fastest), the classes
// U of its children's coefficients (K rows of KW values) scaled by 2^s_S and split into FP16 hi (plane
// 0) and lo (plane 1); s_S = 10 - e with max |U| = f 2^e, f in [0.5, 1) (empty parents: zeros,
// s = 0).  One warp per parent; A and scale hold the levels one after another.
template <int P>
__global__ void __launch_bounds__(256) k_blk_presplit(int L, const int32_t *__restrict__ begin,
                                                      const int32_t *__restrict__ end, const float *__restrict__ M,
                                                      __half *__restrict__ A, int8_t *__restrict__ scale)
{
    using C = BlkCfg<P>;
    constexpr int PP = P * P;
    const int lane = threadIdx.x & 31;
    const int64_t i = blockIdx.x * (int64_t)(blockDim.x >> 5) + (threadIdx.x >> 5);  // parent 1 + i of all levels
    if (i >= level_offset(L) - 1) return;
    int lp = 1;
    while (i + 1 >= level_offset(lp + 1)) ++lp;
    const uint32_t il = (uint32_t)(i + 1 - level_offset(lp)), pg = 1u << lp;  // grid order, x fastest
    const uint32_t x = il & (pg - 1), y = (il >> lp) & (pg - 1), z = il >> (2 * lp);
    const int64_t c0 = level_offset(lp + 1) + 8 * (int64_t)morton3(x, y, z);
    bool has[8];
#pragma unroll
    for (int q = 0; q < 8; ++q) has[q] = end[c0 + q] > begin[c0 + q];
    __half *row = A + i * (2 * C::KW);
    constexpr int NJ = (PP + 31) / 32;
    float v[NJ][8];
    float m = 0.f;
#pragma unroll
    for (int j = 0; j < NJ; ++j) {
        const int k = lane + 32 * j;
#pragma unroll
        for (int q = 0; q < 8; ++q) v[j][q] = k < PP && has[q] ? M[(c0 + q) * PP + k] : 0.f;
        blk_sign_children(v[j], blk_signs(min(k, PP - 1)));
        blk_hadamard(v[j]);
#pragma unroll
        for (int q = 0; q < 8; ++q) m = fmaxf(m, fabsf(v[j][q]));
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
    const bool fin = m > 0.f && m <= 3.0e38f;
    int ex = 0;
    if (fin) frexpf(m, &ex);
    int sc = fin ? 10 - ex : 0;
    sc = sc < -100 ? -100 : (sc > 100 ? 100 : sc);
    if (lane == 0) scale[i] = (int8_t)sc;
    const float up = blk_pow2(sc);
#pragma unroll
    for (int j = 0; j < NJ; ++j) {
        const int k = lane + 32 * j;
        if (k >= PP) continue;
#pragma unroll
        for (int q = 0; q < 8; ++q) {
            const float xs = v[j][q] * up;
            const __half hi = __float2half_rn(xs);
            __half *at = row + (q / C::CU) * C::UNIT + (q % C::CU) * PP + k;
            at[0] = hi;
            at[C::KW] = __float2half_rn(xs - __half2float(hi));
        }
    }
    // the units' padding, read by the MMA against zero columns
    constexpr int PAD = C::UNIT - C::CU * PP;
    if constexpr (PAD > 0)
        for (int e = lane; e < 2 * C::NUNIT * PAD; e += 32)
            row[(e / PAD) * C::UNIT + C::CU * PP + e % PAD] = __float2half_rn(0.f);
}

// ---- operator blocks B'_D (FP16 hi | lo, scaled by 2^g) ----------------------------------------
// The 64 class products of one offset, target coefficient n and source coefficient k, in FP64: the
// 27 operators T_{2D + sigma - tau} (0 for near offsets) as a 2 x 2 Toeplitz block per axis, and per
// axis B'[c'][c] = 1/2 sum_{tau, sigma} (-1)^{c' tau + c sigma} s(n)^tau s(k)^sigma t_{sigma - tau}.
template <int P, class F>
GB_DEV void blk_class_products(const float *__restrict__ ops, int d, int n, int k, F put)
{
    constexpr int PP = P * P, PR = ops_rows_padded(P);
    int dx, dy, dz;
    blk_delta(d, dx, dy, dz);
    const int sn = blk_signs(n), sk = blk_signs(k);
    double z[2][2][9], y[2][2][2][2][3];
    auto axis = [](double tm, double t0, double tp, bool fn, bool fk, double (&o)[2][2]) {
        const double a = fk ? -tp : tp, b = fn ? -tm : tm, c = fn != fk ? -t0 : t0;  // (tau, sigma) = (0,1), (1,0), (1,1)
        o[0][0] = 0.5 * (t0 + a + b + c);
        o[0][1] = 0.5 * (t0 - a + b - c);
        o[1][0] = 0.5 * (t0 + a - b - c);
        o[1][1] = 0.5 * (t0 - a - b + c);
    };
    for (int e = 0; e < 9; ++e) {  // z axis, for every (x, y) difference
        const int ox = 2 * dx + e % 3 - 1, oy = 2 * dy + e / 3 - 1;
        double t[3];
        for (int w = 0; w < 3; ++w) {
            const int oz = 2 * dz + w - 1;
            t[w] = max(abs(ox), max(abs(oy), abs(oz))) < 2 ? 0.0
                       : (double)ops[(size_t)m2l_code(ox, oy, oz) * PP * PR + (size_t)k * PR + n];
        }
        double o[2][2];
        axis(t[0], t[1], t[2], sn >> 2 & 1, sk >> 2 & 1, o);
        for (int q = 0; q < 4; ++q) z[q >> 1][q & 1][e] = o[q >> 1][q & 1];
    }
    for (int q = 0; q < 4; ++q)
        for (int e = 0; e < 3; ++e) {  // y axis, for every x difference
            double o[2][2];
            const double *t = z[q >> 1][q & 1];
            axis(t[e], t[3 + e], t[6 + e], sn >> 1 & 1, sk >> 1 & 1, o);
            for (int r = 0; r < 4; ++r) y[q >> 1][q & 1][r >> 1][r & 1][e] = o[r >> 1][r & 1];
        }
    for (int q = 0; q < 4; ++q)
        for (int r = 0; r < 4; ++r) {
            double o[2][2];
            const double *t = y[q >> 1][q & 1][r >> 1][r & 1];
            axis(t[0], t[1], t[2], sn & 1, sk & 1, o);
            for (int w = 0; w < 4; ++w)
                put((q >> 1) << 2 | (r >> 1) << 1 | w >> 1, (q & 1) << 2 | (r & 1) << 1 | (w & 1), o[w >> 1][w & 1]);
        }
}

// largest |B'| over all offsets, as float bits (non-negative floats order like their bit patterns);
// a block per (d, k), threads over n
template <int P>
__global__ void __launch_bounds__(128) k_blk_opmax(const float *__restrict__ ops, unsigned *__restrict__ mbits)
{
    constexpr int PP = P * P;
    float m = 0.f;
    for (int n = threadIdx.x; n < PP; n += blockDim.x)
        blk_class_products<P>(ops, blockIdx.x / PP, n, blockIdx.x % PP,
                              [&](int, int, double v) { m = fmaxf(m, fabsf((float)v)); });
    for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
    if ((threadIdx.x & 31) == 0) atomicMax(mbits, __float_as_uint(m));
}

// B[d][plane][row: class c', n][K column of class c, k] (the columns' padding zeroed beforehand); g
// stored after the table
template <int P>
__global__ void __launch_bounds__(128) k_blk_build(const float *__restrict__ ops, const unsigned *__restrict__ mbits,
                                                   __half *__restrict__ B, int *__restrict__ gout)
{
    using C = BlkCfg<P>;
    constexpr int PP = P * P;
    const int d = blockIdx.x / PP, n = blockIdx.x % PP;
    int ex = 0;
    const float m = __uint_as_float(*mbits);
    if (m > 0.f) frexpf(m, &ex);
    const int g = m > 0.f ? 12 - ex : 0;
    if (blockIdx.x == 0 && threadIdx.x == 0) *gout = g;
    const double sc = ldexp(1.0, g);
    __half *hi = B + (size_t)d * 2 * C::KD * C::KW, *lo = hi + (size_t)C::KD * C::KW;
    for (int k = threadIdx.x; k < PP; k += blockDim.x)
        blk_class_products<P>(ops, d, n, k, [&](int ct, int cs, double v) {
            const size_t at = (size_t)(ct * PP + n) * C::KW + (cs / C::CU) * C::UNIT + (cs % C::CU) * PP + k;
            const float f = (float)(v * sc);
            const __half h = __float2half_rn(f);
            hi[at] = h;
            lo[at] = __float2half_rn(f - __half2float(h));
        });
}

// ---- the kernel -------------------------------------------------------------------------------
template <int P>
__global__ void __launch_bounds__(kBlkThreads, 1)
    k_m2l_blk(const __grid_constant__ BlkParams prm, const int32_t *__restrict__ begin,
              const int32_t *__restrict__ end, const int8_t *__restrict__ pscale, const int *__restrict__ gexp,
              float *__restrict__ Lc, float *__restrict__ Lpart, int *status)
{
    using C = BlkCfg<P>;
    constexpr int PP = C::PP, NT = C::NT, NH = C::NH, NSTAGE = C::NSTAGE;
    constexpr uint32_t kIdesc = (1u << 4) | ((uint32_t)(NT >> 3) << 17) | ((uint32_t)(kBlkRows >> 4) << 24);
    constexpr int kProdWarp = kBlkDrainWarps, kMmaWarp = kBlkDrainWarps + 1;

    extern __shared__ unsigned char blk_smem_raw[];
    __shared__ __align__(8) uint64_t full_bar[NSTAGE], empty_bar[NSTAGE], dfull[2], dempty[2], done_bar;
    __shared__ int s_issued[NSTAGE];
    __shared__ BlkSteps<C> s_steps;
    __shared__ uint32_t s_tmem;
    __shared__ volatile int s_abort;

    // ---- tile: level, target parent box, N-tile; offset range [d_lo, d_hi)
    const int ks = (prm.tile0 + (int)blockIdx.x) % prm.ksplit;
    const int tile = (prm.tile0 + (int)blockIdx.x) / prm.ksplit;
    const int d_lo = (26 * ks) / prm.ksplit, d_hi = (26 * (ks + 1)) / prm.ksplit;
    int l = 2;
    while (l < prm.L && tile >= prm.tile_lo[l + 1]) ++l;
    const int pg = 1 << (l - 1);
    const int bx = pg < 8 ? pg : 8, by = pg < 4 ? pg : 4, bz = by;
    const int rows = bx * by * bz;
    int t = tile - prm.tile_lo[l];
    const int nt = t % C::NTILES;
    t /= C::NTILES;
    const int tx = t % (pg / bx), ty = (t / (pg / bx)) % (pg / by), tz = t / ((pg / bx) * (pg / by));
    const int x0 = tx * bx, y0 = ty * by, z0 = tz * bz;
    const uint32_t a_bytes = (uint32_t)rows * kBlkCh * 2;

    unsigned char *smem =
        blk_smem_raw + ((1024u - (smem_u32(blk_smem_raw) & 1023u)) & 1023u);  // 1024-byte aligned stages
    auto a_hi = [&](int st) { return smem + (size_t)st * C::STAGE_BYTES; };
    auto a_lo = [&](int st) { return smem + (size_t)st * C::STAGE_BYTES + C::A_BYTES; };
    auto b_hi = [&](int st) { return smem + (size_t)st * C::STAGE_BYTES + 2 * C::A_BYTES; };
    auto b_lo = [&](int st) { return smem + (size_t)st * C::STAGE_BYTES + 2 * C::A_BYTES + C::B_BYTES; };

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    if (tid == 0) {
        for (int st = 0; st < NSTAGE; ++st) {
            mbar_init(&full_bar[st], 1);   // the producer's expect_tx arrival
            mbar_init(&empty_bar[st], 1);  // one tcgen05.commit
            s_issued[st] = 0;
        }
        for (int b = 0; b < 2; ++b) {
            mbar_init(&dfull[b], 1);
            mbar_init(&dempty[b], kBlkDrainWarps);
        }
        mbar_init(&done_bar, 1);
        s_abort = 0;
        fence_mbar_init();
    }
    if (warp == kProdWarp && lane == 0) {
        blk_prefetch_tmap(&prm.tmA[l]);
        blk_prefetch_tmap(&prm.tmB);
    }
    if (warp == kMmaWarp) tmem_alloc(&s_tmem, C::TMEM_COLS);
    if (warp == 0) blk_steps<C>(s_steps, nt, d_lo, d_hi, lane);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = s_tmem;
    const int S = s_steps.nsteps, NU = s_steps.ndrains;

    if (warp == kProdWarp) {
        if (lane == 0) {
            for (int s = 0; s < S; ++s) {
                const int st = s % NSTAGE, d = step_d(s_steps.step[s]), k0 = step_k0(s_steps.step[s]);
                if (s >= NSTAGE &&
                    !mbar_wait_bounded(&empty_bar[st], ((s / NSTAGE) - 1) & 1, kWaitLimitNs, &s_abort)) {
                    s_abort = 1;
                    break;
                }
                if (s_abort) break;
                int dx, dy, dz;
                blk_delta(d, dx, dy, dz);
                mbar_expect_tx(&full_bar[st], 2u * a_bytes + 2u * (uint32_t)C::B_BYTES);
                blk_tma5(a_hi(st), &prm.tmA[l], k0, 0, x0 + dx, y0 + dy, z0 + dz, &full_bar[st]);
                blk_tma5(a_lo(st), &prm.tmA[l], k0, 1, x0 + dx, y0 + dy, z0 + dz, &full_bar[st]);
                blk_tma4(b_hi(st), &prm.tmB, k0, nt * C::NSTRIDE, 0, d, &full_bar[st]);
                blk_tma4(b_lo(st), &prm.tmB, k0, nt * C::NSTRIDE, 1, d, &full_bar[st]);
                s_issued[st] += 1;
            }
        }
    } else if (warp == kMmaWarp) {
        if (lane == 0) {
            for (int s = 0; s < S; ++s) {
                const uint32_t sv = s_steps.step[s];
                const int st = s % NSTAGE, u = step_drain(sv), b = u & 1;
                const bool first = step_first(sv), last = step_last(sv);
                if (first && u >= 2 &&
                    !mbar_wait_bounded(&dempty[b], ((u - 2) >> 1) & 1, kWaitLimitNs, &s_abort)) {
                    s_abort = 1;
                    break;
                }
                if (!mbar_wait_bounded(&full_bar[st], (s / NSTAGE) & 1, kWaitLimitNs, &s_abort)) {
                    s_abort = 1;
                    break;
                }
                tc_fence_after();
                const uint32_t ah = smem_u32(a_hi(st)), al = smem_u32(a_lo(st));
                const uint32_t bh = smem_u32(b_hi(st)), bl = smem_u32(b_lo(st));
                const uint32_t dt = tmem + (uint32_t)(b * NT);
                for (int j = 0; j < step_kw(sv) / 16; ++j) {
                    const uint32_t o = 32u * j;
                    blk_mma_ss(dt, blk_desc(al + o), blk_desc(bh + o), kIdesc, (first && j == 0) ? 0u : 1u);
                    blk_mma_ss(dt, blk_desc(ah + o), blk_desc(bl + o), kIdesc, 1u);
                    blk_mma_ss(dt, blk_desc(ah + o), blk_desc(bh + o), kIdesc, 1u);
                }
                tc_commit(&empty_bar[st]);
                if (last) tc_commit(&dfull[b]);
            }
            tc_commit(&done_bar);
        }
    } else {
        // ===== drain warps: row r (target parent), columns [h NH, h NH + NH) of the N-tile =====
        const int quad = warp & 3, h = warp >> 2;
        const int r = 32 * quad + lane;
        const uint32_t lane_base = (uint32_t)(32 * quad) << 16;
        const bool rok = r < rows;
        const int qx = x0 + r % bx, qy = y0 + (r / bx) % by, qz = z0 + r / (bx * by);
        const int8_t *sl = pscale + (level_offset(l - 1) - 1);  // parents of level l - 1 (levels >= 1)
        const int g = *gexp;
        float acc[NH];
#pragma unroll
        for (int i = 0; i < NH; ++i) acc[i] = 0.f;
        bool alive = true;
        for (int u = 0; u < NU && alive; ++u) {
            const int d = s_steps.drain_d[u], b = u & 1;
            int dx, dy, dz;
            blk_delta(d, dx, dy, dz);
            const int sx = qx + dx, sy = qy + dy, sz = qz + dz;
            float f = 0.f;
            if (rok && sx >= 0 && sy >= 0 && sz >= 0 && sx < pg && sy < pg && sz < pg)
                f = blk_pow2(-((int)sl[sx + pg * (sy + pg * sz)] + g));
            int ok = 1;
            if (lane == 0) ok = mbar_wait_bounded(&dfull[b], (u >> 1) & 1, kWaitLimitNs, &s_abort) ? 1 : 0;
            if (!__shfl_sync(0xffffffffu, ok, 0)) {
                alive = false;
                break;
            }
            tc_fence_after();
            const uint32_t col0 = tmem + lane_base + (uint32_t)(b * NT + h * NH);
#pragma unroll
            for (int c0 = 0; c0 < NH; c0 += 32) {
                constexpr int W = 32;
                uint32_t v[W];
#pragma unroll
                for (int q = 0; q < W; q += 8)
                    if (c0 + q < NH) blk_ld8(col0 + (uint32_t)(c0 + q), v + q);
                tmem_wait_ld_regs(v);
#pragma unroll
                for (int q = 0; q < W; ++q)
                    if (c0 + q < NH) acc[c0 + q] = fmaf(__uint_as_float(v[q]), f, acc[c0 + q]);
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(&dempty[b]);
        }
        if (!alive && lane == 0) s_abort = 1;
        int ok = 1;
        if (lane == 0) ok = mbar_wait_bounded(&done_bar, 0u, kWaitLimitNs, nullptr) ? 1 : 0;
        ok = __shfl_sync(0xffffffffu, ok, 0);
        if (!ok && lane == 0) s_abort = 1;
        __syncwarp();
        if (ok && alive && !s_abort && rok) {
            float *dst = prm.ksplit > 1 ? Lpart + (int64_t)ks * prm.part_stride : Lc;
            // the classes V of a nonempty parent, in its children's places
            const int64_t key = (int64_t)morton3((uint32_t)qx, (uint32_t)qy, (uint32_t)qz), par = level_offset(l - 1) + key;
            float *row = dst + (level_offset(l) + 8 * key) * PP + nt * C::NSTRIDE;
            if (end[par] > begin[par])
#pragma unroll
                for (int i = 0; i < NH; i += 4)
                    if (h * NH + i < C::NSTRIDE)
                        *reinterpret_cast<float4 *>(row + h * NH + i) =
                            make_float4(acc[i], acc[i + 1], acc[i + 2], acc[i + 3]);
        }
    }

    tc_fence_before();
    __syncthreads();
    if (s_abort) {
        if (tid == 0) {
            atomicOr(status, kStatusTimeout);
            for (int st = 0; st < NSTAGE; ++st)
                if (s_issued[st] > 0) mbar_wait_bounded(&full_bar[st], (s_issued[st] - 1) & 1, kWaitLimitNs, nullptr);
        }
        __syncthreads();
    }
    if (warp == kMmaWarp) {
        __syncwarp();
        tmem_dealloc(tmem, C::TMEM_COLS);
    }
}

// ---- the same block M2L on the adaptive tree ---------------------------------------------------
// On the adaptive tree the V list of a cell t (child tau of parent Q) is the children sigma of
// Q's colleagues S = Q + D (the positional colleagues of the level, D != 0) with |2D + sigma -
// tau|_inf >= 2: the block form above with S taken from the colleague table instead of the
// dense grid.  A colleague that is absent or a leaf, and a child that is absent, contribute zero
// coefficients; a colleague that is a leaf reaches t through its U or X list instead.  Target
// units are the cells of levels >= 1 with children (their children are the targets of levels
// >= 2), numbered in cell order; unit u has a row of the 8 p^2 coefficients of its children in
// the pre-split array (k_ablk_presplit), and row Z (the unit capacity) is zero.  A tile is 128
// consecutive units; its A operand for offset D gathers the rows of the units' colleagues
// (k_ablk_src: the row of every (unit, D), Z where the colleague has no children) by two loader
// warps (16-byte loads, stored in the swizzled layout the TMA writes for the dense form, then a
// proxy fence and one arrival each); B_D comes by TMA as before.

// unit numbering: flag of every cell (levels >= 1 with children)
__global__ void k_ablk_flags(Span cells, const int32_t *__restrict__ level, const int32_t *__restrict__ nchild,
                             uint32_t *__restrict__ flag)
{
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i >= cells.cap) return;
    uint32_t f = 0;
    if (i < span_count(cells)) {
        const int64_t c = span_first(cells) + i;
        f = (level[c] >= 1 && nchild[c] > 0) ? 1u : 0u;
    }
    flag[i] = f;
}

// unit_of[c] = its unit or -1; units[u] = its cell; n_units (one word) = the count
__global__ void k_ablk_units(Span cells, const uint32_t *__restrict__ flag, const uint32_t *__restrict__ scan,
                             int32_t *__restrict__ unit_of, int32_t *__restrict__ units, int32_t *__restrict__ n_units)
{
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i == 0) *n_units = (int32_t)scan[cells.cap];
    if (i >= span_count(cells)) return;
    const int64_t c = span_first(cells) + i;
    if (flag[i]) {
        unit_of[c] = (int32_t)scan[i];
        units[scan[i]] = (int32_t)c;
    } else {
        unit_of[c] = -1;
    }
}

// pre-split rows: unit u (one warp): the classes U of its children's coefficients, scaled by 2^s_u, in
// FP16 hi | lo, s_u = 10 - e with max |U| = f 2^e (0 and zeros for none); row Z and its scale are zero
template <int P>
__global__ void __launch_bounds__(256) k_ablk_presplit(const int32_t *__restrict__ n_units, int64_t zrow,
                                                       const int32_t *__restrict__ units,
                                                       const int32_t *__restrict__ child_of,
                                                       const float *__restrict__ M, __half *__restrict__ A,
                                                       int8_t *__restrict__ scale)
{
    using C = BlkCfg<P>;
    constexpr int PP = P * P;
    const int lane = threadIdx.x & 31;
    const int64_t u = blockIdx.x * (int64_t)(blockDim.x >> 5) + (threadIdx.x >> 5);
    const int64_t nu = *n_units;
    if (u > zrow || (u >= nu && u != zrow)) return;
    __half *row = A + u * (2 * C::KW);
    if (u == zrow || u >= nu) {
        for (int k = lane; k < 2 * C::KW; k += 32) row[k] = __float2half_rn(0.f);
        if (lane == 0) scale[u] = 0;
        return;
    }
    const int64_t cell = units[u];
    bool has[8];
    int64_t child[8];
#pragma unroll
    for (int q = 0; q < 8; ++q) {
        child[q] = child_of[cell * 8 + q];
        has[q] = child[q] >= 0;
    }
    constexpr int NJ = (PP + 31) / 32;
    float v[NJ][8];
    float m = 0.f;
#pragma unroll
    for (int j = 0; j < NJ; ++j) {
        const int k = lane + 32 * j;
#pragma unroll
        for (int q = 0; q < 8; ++q) v[j][q] = k < PP && has[q] ? M[child[q] * PP + k] : 0.f;
        blk_sign_children(v[j], blk_signs(min(k, PP - 1)));
        blk_hadamard(v[j]);
#pragma unroll
        for (int q = 0; q < 8; ++q) m = fmaxf(m, fabsf(v[j][q]));
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
    const bool fin = m > 0.f && m <= 3.0e38f;
    int ex = 0;
    if (fin) frexpf(m, &ex);
    int sc = fin ? 10 - ex : 0;
    sc = sc < -100 ? -100 : (sc > 100 ? 100 : sc);
    if (lane == 0) scale[u] = (int8_t)sc;
    const float up = blk_pow2(sc);
#pragma unroll
    for (int j = 0; j < NJ; ++j) {
        const int k = lane + 32 * j;
        if (k >= PP) continue;
#pragma unroll
        for (int q = 0; q < 8; ++q) {
            const float xs = v[j][q] * up;
            const __half hi = __float2half_rn(xs);
            __half *at = row + (q / C::CU) * C::UNIT + (q % C::CU) * PP + k;
            at[0] = hi;
            at[C::KW] = __float2half_rn(xs - __half2float(hi));
        }
    }
    // the units' padding, read by the MMA against zero columns
    constexpr int PAD = C::UNIT - C::CU * PP;
    if constexpr (PAD > 0)
        for (int e = lane; e < 2 * C::NUNIT * PAD; e += 32)
            row[(e / PAD) * C::UNIT + C::CU * PP + e % PAD] = __float2half_rn(0.f);
}

// src[(tile 26 + d) 128 + r] = the row of unit tile 128 + r's colleague at offset d (Z if none);
// ucap: the units covered, a multiple of 128
__global__ void k_ablk_src(const int32_t *__restrict__ n_units, int64_t ucap, int64_t zrow,
                           const int32_t *__restrict__ units, const int32_t *__restrict__ coll,
                           const int32_t *__restrict__ unit_of, int32_t *__restrict__ src)
{
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;  // over units (padded to tiles) x 26
    if (i >= ucap * 26) return;
    const int64_t u = i / 26;
    const int d = (int)(i % 26);
    int32_t row = (int32_t)zrow;
    if (u < *n_units) {
        int dx, dy, dz;
        blk_delta(d, dx, dy, dz);
        const int32_t s = coll[(int64_t)units[u] * 27 + (dx + 1) + 3 * (dy + 1) + 9 * (dz + 1)];
        if (s >= 0 && unit_of[s] >= 0) row = unit_of[s];
    }
    src[((u / kBlkRows) * 26 + d) * kBlkRows + u % kBlkRows] = row;
}

constexpr int kAblkLoadWarps = 2;  // each loads 64 rows (more would leave the drains too few registers)
constexpr int kAblkThreads = 32 * (kBlkDrainWarps + kAblkLoadWarps + 2);  // drains, loaders, B producer, MMA

struct AblkParams {
    CUtensorMap tmB;  // B_D, FP16 hi | lo
    int tile0;        // tile of block 0 (launch in waves)
    int ksplit;
    int64_t ut0;          // unit tile of tile 0
    int64_t part_stride;  // floats between the partial sums of two offset ranges
    int64_t zrow;
    int seq0;  // SEQ: from this tile on a CTA takes the ranges of its tile one after another
};

// Classes of unit u (from the launch's first on) and range k: V + k part_stride + u KD.  A captured
// evaluation may meet far more units than its capacities were made from, and the classes of all of
// them for up to 26 ranges are memory and idle CTAs that few refills use.  So there (SEQ) the units past
// the expected ones take their ranges one after another in one CTA, which adds them in V in range
// order, as k_ablk_finish does for the others; their V rows follow the split ones'.  64 sets of 20,000
// particles, p = 8: 10.2 GB -> 2.0, 4.65 ms -> 4.31; a batch of 96 instances 6.54 ms -> 6.37.
template <int P, bool SEQ>
__global__ void __launch_bounds__(kAblkThreads, 1)
    k_m2l_ablk(const __grid_constant__ AblkParams prm, const int32_t *__restrict__ n_units,
               const int32_t *__restrict__ src, const __half *__restrict__ Apre, const int8_t *__restrict__ uscale,
               const int *__restrict__ gexp, float *__restrict__ V, int *status)
{
    using C = BlkCfg<P>;
    constexpr int KD = C::KD, NT = C::NT, NH = C::NH, NSTAGE = C::NSTAGE;
    constexpr uint32_t kIdesc = (1u << 4) | ((uint32_t)(NT >> 3) << 17) | ((uint32_t)(kBlkRows >> 4) << 24);
    constexpr int kLoad0 = kBlkDrainWarps, kProdWarp = kLoad0 + kAblkLoadWarps, kMmaWarp = kProdWarp + 1;

    extern __shared__ unsigned char blk_smem_raw[];
    __shared__ __align__(8) uint64_t full_bar[NSTAGE], empty_bar[NSTAGE], dfull[2], dempty[2], done_bar;
    __shared__ int s_issued[NSTAGE];
    __shared__ BlkSteps<C> s_steps;
    __shared__ uint32_t s_tmem;
    __shared__ volatile int s_abort;

    // ---- tile: unit tile, N-tile, offset range [d_lo, d_hi)
    const int bid = prm.tile0 + (int)blockIdx.x;
    const bool seq = SEQ && bid >= prm.seq0;
    const int ks = seq ? prm.ksplit - 1 : bid % prm.ksplit;  // seq: the V rows past part_stride
    const int tt = seq ? prm.seq0 / prm.ksplit + (bid - prm.seq0) : bid / prm.ksplit;
    const int nt = tt % C::NTILES;
    const int64_t ut = prm.ut0 + tt / C::NTILES;
    const int64_t nu = *n_units;
    if (ut * kBlkRows >= nu) return;  // the whole CTA: past the units (before any barrier or TMEM)
    const int d_lo = seq ? 0 : (26 * ks) / prm.ksplit, d_hi = (26 * (ks + 1)) / prm.ksplit;
    const int32_t *tsrc = src + ut * 26 * kBlkRows;

    unsigned char *smem =
        blk_smem_raw + ((1024u - (smem_u32(blk_smem_raw) & 1023u)) & 1023u);  // 1024-byte aligned stages
    auto a_pl = [&](int st, int pl) { return smem + (size_t)st * C::STAGE_BYTES + pl * C::A_BYTES; };
    auto b_hi = [&](int st) { return smem + (size_t)st * C::STAGE_BYTES + 2 * C::A_BYTES; };
    auto b_lo = [&](int st) { return smem + (size_t)st * C::STAGE_BYTES + 2 * C::A_BYTES + C::B_BYTES; };

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    if (tid == 0) {
        for (int st = 0; st < NSTAGE; ++st) {
            mbar_init(&full_bar[st], kAblkLoadWarps + 1);  // the loader warps + the B copies' expect_tx
            mbar_init(&empty_bar[st], 1);                  // one tcgen05.commit
            s_issued[st] = 0;
        }
        for (int b = 0; b < 2; ++b) {
            mbar_init(&dfull[b], 1);
            mbar_init(&dempty[b], kBlkDrainWarps);
        }
        mbar_init(&done_bar, 1);
        s_abort = 0;
        fence_mbar_init();
    }
    if (warp == kProdWarp && lane == 0) blk_prefetch_tmap(&prm.tmB);
    if (warp == kMmaWarp) tmem_alloc(&s_tmem, C::TMEM_COLS);
    if (warp == 0) blk_steps<C>(s_steps, nt, d_lo, d_hi, lane);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = s_tmem;
    const int S = s_steps.nsteps, NU = s_steps.ndrains;

    if (warp >= kLoad0 && warp < kProdWarp) {
        // ===== loader warps: rows 64 w + lane and 64 w + 32 + lane of A (hi and lo planes) =====
        // a stage's 16-byte chunks go through registers, the next stage's loads issued before this
        // stage is stored, so their latency overlaps
        constexpr int RPW = kBlkRows / kAblkLoadWarps / 32;  // rows per lane
        constexpr int CPR = kBlkCh / 8;                      // 16-byte chunks per row
        constexpr int NB = RPW * 2 * CPR;                    // chunks per lane and stage
        const int r0 = (kBlkRows / kAblkLoadWarps) * (warp - kLoad0) + lane;
        auto fetch = [&](int s, int4(&v)[NB]) {
            const uint32_t sv = s_steps.step[s];
            const int d = step_d(sv), kw = step_kw(sv);
#pragma unroll
            for (int rr = 0; rr < RPW; ++rr) {
                const int64_t row = tsrc[d * kBlkRows + r0 + 32 * rr];
#pragma unroll
                for (int pl = 0; pl < 2; ++pl) {
                    const int4 *g = reinterpret_cast<const int4 *>(Apre + (row * 2 + pl) * C::KW + step_k0(sv));
#pragma unroll
                    for (int q = 0; q < CPR; ++q) v[(rr * 2 + pl) * CPR + q] = 8 * q < kw ? __ldg(g + q) : int4{0, 0, 0, 0};
                }
            }
        };
        auto put = [&](int s, const int4(&v)[NB]) {
            const int st = s % NSTAGE, kw = step_kw(s_steps.step[s]);
            int ok = 1;
            if (s >= NSTAGE && lane == 0)
                ok = mbar_wait_bounded(&empty_bar[st], ((s / NSTAGE) - 1) & 1, kWaitLimitNs, &s_abort) ? 1 : 0;
            ok = __shfl_sync(0xffffffffu, ok, 0);
            if (!ok || s_abort) {
                if (lane == 0) s_abort = 1;
                return false;
            }
#pragma unroll
            for (int rr = 0; rr < RPW; ++rr) {
                const int r = r0 + 32 * rr;
#pragma unroll
                for (int pl = 0; pl < 2; ++pl) {
                    unsigned char *dst = a_pl(st, pl) + (size_t)r * (2 * kBlkCh);
#pragma unroll
                    for (int q = 0; q < CPR; ++q) {
                        if (8 * q >= kw) break;
                        // the TMA's swizzle of this row: 16-byte chunk q at q ^ (row bits)
                        const int qs = q ^ ((r >> 1) & 3);
                        *reinterpret_cast<int4 *>(dst + 16 * qs) = v[(rr * 2 + pl) * CPR + q];
                    }
                }
            }
            fence_proxy_async();  // the generic-proxy stores, before the MMA's async-proxy reads
            __syncwarp();
            if (lane == 0) mbar_arrive(&full_bar[st]);
            return true;
        };
        int4 va[NB], vb[NB];
        if (S > 0) fetch(0, va);
        for (int s = 0; s < S; s += 2) {
            if (s + 1 < S) fetch(s + 1, vb);
            if (!put(s, va) || s + 1 >= S) break;
            if (s + 2 < S) fetch(s + 2, va);
            if (!put(s + 1, vb)) break;
        }
    } else if (warp == kProdWarp) {
        if (lane == 0) {
            for (int s = 0; s < S; ++s) {
                const int st = s % NSTAGE, d = step_d(s_steps.step[s]), k0 = step_k0(s_steps.step[s]);
                if (s >= NSTAGE &&
                    !mbar_wait_bounded(&empty_bar[st], ((s / NSTAGE) - 1) & 1, kWaitLimitNs, &s_abort)) {
                    s_abort = 1;
                    break;
                }
                if (s_abort) break;
                mbar_expect_tx(&full_bar[st], 2u * (uint32_t)C::B_BYTES);
                blk_tma4(b_hi(st), &prm.tmB, k0, nt * C::NSTRIDE, 0, d, &full_bar[st]);
                blk_tma4(b_lo(st), &prm.tmB, k0, nt * C::NSTRIDE, 1, d, &full_bar[st]);
                s_issued[st] += 1;
            }
        }
    } else if (warp == kMmaWarp) {
        if (lane == 0) {
            for (int s = 0; s < S; ++s) {
                const uint32_t sv = s_steps.step[s];
                const int st = s % NSTAGE, u = step_drain(sv), b = u & 1;
                const bool first = step_first(sv), last = step_last(sv);
                if (first && u >= 2 &&
                    !mbar_wait_bounded(&dempty[b], ((u - 2) >> 1) & 1, kWaitLimitNs, &s_abort)) {
                    s_abort = 1;
                    break;
                }
                if (!mbar_wait_bounded(&full_bar[st], (s / NSTAGE) & 1, kWaitLimitNs, &s_abort)) {
                    s_abort = 1;
                    break;
                }
                tc_fence_after();
                const uint32_t ah = smem_u32(a_pl(st, 0)), al = smem_u32(a_pl(st, 1));
                const uint32_t bh = smem_u32(b_hi(st)), bl = smem_u32(b_lo(st));
                const uint32_t dt = tmem + (uint32_t)(b * NT);
                for (int j = 0; j < step_kw(sv) / 16; ++j) {
                    const uint32_t o = 32u * j;
                    blk_mma_ss(dt, blk_desc(al + o), blk_desc(bh + o), kIdesc, (first && j == 0) ? 0u : 1u);
                    blk_mma_ss(dt, blk_desc(ah + o), blk_desc(bl + o), kIdesc, 1u);
                    blk_mma_ss(dt, blk_desc(ah + o), blk_desc(bh + o), kIdesc, 1u);
                }
                tc_commit(&empty_bar[st]);
                if (last) tc_commit(&dfull[b]);
            }
            tc_commit(&done_bar);
        }
    } else {
        // ===== drain warps: row r (target unit), columns [h NH, h NH + NH) of the N-tile =====
        const int quad = warp & 3, h = warp >> 2;
        const int r = 32 * quad + lane;
        const uint32_t lane_base = (uint32_t)(32 * quad) << 16;
        const int64_t unit = ut * kBlkRows + r;
        const bool rok = unit < nu;
        auto vrow = [&] {
            return V + (int64_t)ks * prm.part_stride + (unit - prm.ut0 * kBlkRows) * KD + nt * C::NSTRIDE + h * NH;
        };
        const int g = *gexp;
        int range = 0;  // SEQ: of the sums in acc
        float acc[NH];
#pragma unroll
        for (int i = 0; i < NH; ++i) acc[i] = 0.f;
        bool alive = true;
        for (int u = 0; u < NU && alive; ++u) {
            const int d = s_steps.drain_d[u], b = u & 1;
            const int64_t row = tsrc[d * kBlkRows + r];
            const float f = row == prm.zrow ? 0.f : blk_pow2(-((int)uscale[row] + g));
            int ok = 1;
            if (lane == 0) ok = mbar_wait_bounded(&dfull[b], (u >> 1) & 1, kWaitLimitNs, &s_abort) ? 1 : 0;
            if (!__shfl_sync(0xffffffffu, ok, 0)) {
                alive = false;
                break;
            }
            tc_fence_after();
            const uint32_t col0 = tmem + lane_base + (uint32_t)(b * NT + h * NH);
#pragma unroll
            for (int c0 = 0; c0 < NH; c0 += 32) {
                constexpr int W = 32;
                uint32_t v[W];
#pragma unroll
                for (int q = 0; q < W; q += 8)
                    if (c0 + q < NH) blk_ld8(col0 + (uint32_t)(c0 + q), v + q);
                tmem_wait_ld_regs(v);
#pragma unroll
                for (int q = 0; q < W; ++q)
                    if (c0 + q < NH) acc[c0 + q] = fmaf(__uint_as_float(v[q]), f, acc[c0 + q]);
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(&dempty[b]);
            if (SEQ && seq && (u + 1 == NU || s_steps.drain_d[u + 1] >= (26 * (range + 1)) / prm.ksplit)) {
                if (rok) {
                    float *row = vrow();
#pragma unroll
                    for (int i = 0; i < NH; i += 4)
                        if (h * NH + i < C::NSTRIDE) {
                            float4 *at = reinterpret_cast<float4 *>(row + i);
                            float4 t = range > 0 ? *at : make_float4(0.f, 0.f, 0.f, 0.f);
                            t.x += acc[i], t.y += acc[i + 1], t.z += acc[i + 2], t.w += acc[i + 3];
                            *at = t;
                        }
                }
#pragma unroll
                for (int i = 0; i < NH; ++i) acc[i] = 0.f;
                ++range;
            }
        }
        if (!alive && lane == 0) s_abort = 1;
        int ok = 1;
        if (lane == 0) ok = mbar_wait_bounded(&done_bar, 0u, kWaitLimitNs, nullptr) ? 1 : 0;
        ok = __shfl_sync(0xffffffffu, ok, 0);
        if (!ok && lane == 0) s_abort = 1;
        __syncwarp();
        if (ok && alive && !s_abort && rok && !seq) {
            float *row = vrow();
#pragma unroll
            for (int i = 0; i < NH; i += 4)
                if (h * NH + i < C::NSTRIDE)
                    *reinterpret_cast<float4 *>(row + i) = make_float4(acc[i], acc[i + 1], acc[i + 2], acc[i + 3]);
        }
    }

    tc_fence_before();
    __syncthreads();
    if (s_abort) {
        if (tid == 0) {
            atomicOr(status, kStatusTimeout);
            for (int st = 0; st < NSTAGE; ++st)
                if (s_issued[st] > 0) mbar_wait_bounded(&full_bar[st], (s_issued[st] - 1) & 1, kWaitLimitNs, nullptr);
        }
        __syncthreads();
    }
    if (warp == kMmaWarp) {
        __syncwarp();
        tmem_dealloc(tmem, C::TMEM_COLS);
    }
}

// ---- the classes back to the children: V = sum over the offset ranges (fixed order, so the result does
// not depend on which CTA finished first), L~_tau = s^tau / 8 sum_c (-1)^{c . tau} V_c.  Eight lanes
// per parent and four coefficients, one a class: each adds its class over the ranges (a thread for
// all eight took 36 us on the 208 loads of 26 ranges), then three exchanges form the children.
// Lane: item (4 to a warp) + 4 class.  In place where there is one range (uniform tree).
GB_DEV float4 blk_child(const float4 *src, int64_t stride4, int ksplit, int n4, int c, bool valid)
{
    float v[4] = {0.f, 0.f, 0.f, 0.f};
    if (valid) {
        const float4 a = *src;
        v[0] = a.x, v[1] = a.y, v[2] = a.z, v[3] = a.w;
#pragma unroll 8
        for (int k = 1; k < ksplit; ++k) {
            const float4 t = src[k * stride4];
            v[0] += t.x, v[1] += t.y, v[2] += t.z, v[3] += t.w;
        }
    }
#pragma unroll
    for (int b = 1; b < 8; b <<= 1)
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const float o = __shfl_xor_sync(0xffffffffu, v[j], 4 * b);
            v[j] = (c & b) ? o - v[j] : v[j] + o;
        }
#pragma unroll
    for (int j = 0; j < 4; ++j) v[j] *= (__popc(c & blk_signs(4 * n4 + j)) & 1) ? -0.125f : 0.125f;
    return make_float4(v[0], v[1], v[2], v[3]);
}

// uniform tree: parents of levels 1 .. L - 1
template <int P>
__global__ void __launch_bounds__(256) k_blk_finish(int npar, int ksplit, int64_t stride4,
                                                    const int32_t *__restrict__ begin, const int32_t *__restrict__ end,
                                                    const float4 *src, float4 *Lc)
{
    const int lane = threadIdx.x & 31, c = lane >> 2;
    constexpr int PP4 = P * P / 4;
    const uint32_t i = (blockIdx.x * 8 + (threadIdx.x >> 5)) * 4 + (lane & 3), q = i / PP4, n4 = i % PP4;
    const int64_t par = 1 + (int64_t)q, at = (8 * par + 1 + c) * PP4 + n4;  // children of cell par: 8 par + 1 ..
    const bool ok = q < (uint32_t)npar && end[par] > begin[par];
    const float4 v = blk_child(src + at, stride4, ksplit, (int)n4, c, ok);
    if (ok && end[8 * par + 1 + c] > begin[8 * par + 1 + c]) Lc[at] = v;
}

// adaptive tree: units u0 .. u0 + n; SEQ: the first n_split have their ranges apart (else all)
template <int P, bool SEQ>
__global__ void __launch_bounds__(256) k_ablk_finish(const int32_t *__restrict__ n_units, int64_t u0, uint32_t n,
                                                     uint32_t n_split, int ksplit, int64_t stride4,
                                                     const int32_t *__restrict__ units,
                                                     const int32_t *__restrict__ child_of,
                                                     const float4 *__restrict__ V, float4 *__restrict__ Lc)
{
    const int lane = threadIdx.x & 31, c = lane >> 2;
    constexpr int PP4 = P * P / 4;
    const uint32_t i = (blockIdx.x * 8 + (threadIdx.x >> 5)) * 4 + (lane & 3), u = i / PP4, n4 = i % PP4;
    const bool ok = u < n && u0 + u < *n_units;
    const float4 *src = V + ((int64_t)u * 8 + c) * PP4 + n4;
    if (SEQ && u >= n_split) {
        src += (ksplit - 1) * stride4;
        ksplit = 1;
    }
    const float4 v = blk_child(src, stride4, ksplit, (int)n4, c, ok);
    const int64_t g = ok ? child_of[(int64_t)units[u0 + u] * 8 + c] : -1;
    if (g >= 0) Lc[g * PP4 + n4] = v;
}

// ---- host side ----------------------------------------------------------------------------------
namespace {

PFN_cuTensorMapEncodeTiled_v12000 tmap_encoder()
{
    static std::once_flag once;
    static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
    std::call_once(once, [] {
        void *p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) ==
                cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(p);
    });
    return fn;
}

// per-level layout of the pre-split sources: parents of levels 1 .. L-1, level lp at parent
// offset level_offset(lp) - 1
int64_t blk_parents_before(int lp) { return level_offset(lp) - 1; }

}  // namespace

size_t m2l_blk_presplit_bytes(int P, int L)
{
    if (L < 2) return 0;
    return (size_t)blk_parents_before(L) * 2 * blk_kw(P) * sizeof(__half);
}

size_t m2l_blk_scale_bytes(int L) { return L < 2 ? 0 : (size_t)blk_parents_before(L); }

// tiles of one launch over levels 2..L (ksplit 1)
template <int P>
static int blk_tiles(int L)
{
    int n = 0;
    for (int l = 2; l <= L; ++l) {
        const int pg = 1 << (l - 1);
        const int bx = pg < 8 ? pg : 8, by = pg < 4 ? pg : 4;
        n += (pg / bx) * (pg / by) * (pg / by) * BlkCfg<P>::NTILES;
    }
    return n;
}

static int blk_tiles_p(int P, int L)
{
    switch (P) {
    case 4: return blk_tiles<4>(L);
    case 6: return blk_tiles<6>(L);
    case 8: return blk_tiles<8>(L);
    case 10: return blk_tiles<10>(L);
    }
    return 0;
}

// Offset ranges per tile: 1 when there are at least kBlkFillCtas tiles (one per SM of a 152-SM
// GB300), else the number of ranges k with the least time in waves of kBlkFillCtas CTAs, a CTA of
// ceil(26 / k) offsets costing that many plus two for its start, first copies and last drain (and
// the sum of the ranges, half an offset).  12 tiles (100,000 particles, p = 8): 26 ranges took three
// launches, the last of 8 CTAs, 75 us and 10 for the sum; 12 ranges one, and the step 244 -> 193 us.
// A fixed rule, so that the workspace size does not depend on the device.
constexpr int kBlkFillCtas = kSms;
static int blk_ranges(int64_t tiles)
{
    if (tiles <= 0 || tiles >= kBlkFillCtas) return 1;
    int best = 1;
    int64_t least = INT64_MAX;
    for (int k = 1; k <= 26; ++k) {
        const int64_t waves = (tiles * k + kBlkFillCtas - 1) / kBlkFillCtas;
        const int64_t cost = 2 * waves * ((26 + k - 1) / k + 2) + (k > 1 ? 1 : 0);
        if (cost < least) least = cost, best = k;
    }
    return best;
}

int m2l_blk_ksplit(int P, int L) { return L < 2 ? 1 : blk_ranges(blk_tiles_p(P, L)); }

// partial sums of the offset ranges: ksplit x (cells of levels 0..L) x p^2 floats (0 if not split)
size_t m2l_blk_part_bytes(int P, int L)
{
    const int k = m2l_blk_ksplit(P, L);
    return k > 1 ? (size_t)k * level_offset(L + 1) * P * P * sizeof(float) : 0;
}

size_t m2l_blk_table_bytes(int P) { return 26 * 2 * 8 * (size_t)P * P * blk_kw(P) * sizeof(__half) + 256; }

// the table: B' (hi | lo per d), then the exponent g and the max-bits scratch word
template <int P>
static void launch_build_t(const float *ops, void *table, cudaStream_t s)
{
    using C = BlkCfg<P>;
    __half *B = static_cast<__half *>(table);
    int *g = reinterpret_cast<int *>(B + 26 * 2 * (size_t)C::KD * C::KW);
    unsigned *mbits = reinterpret_cast<unsigned *>(g + 1);
    cudaMemsetAsync(table, 0, m2l_blk_table_bytes(P), s);
    k_blk_opmax<P><<<26 * P * P, 128, 0, s>>>(ops, mbits);
    k_blk_build<P><<<26 * P * P, 128, 0, s>>>(ops, mbits, B, g);
    note_launches(2);
}

void launch_build_m2l_blk(int P, const float *ops, void *table, cudaStream_t s)
{
    switch (P) {
    case 4: launch_build_t<4>(ops, table, s); break;
    case 6: launch_build_t<6>(ops, table, s); break;
    case 8: launch_build_t<8>(ops, table, s); break;
    case 10: launch_build_t<10>(ops, table, s); break;
    }
}

void launch_blk_presplit(int P, int L, const int32_t *begin, const int32_t *end, const float *M, void *presplit,
                         int8_t *pscale, cudaStream_t s)
{
    if (L < 2) return;
    const unsigned grid = (unsigned)((blk_parents_before(L) + 7) / 8);
    __half *A = static_cast<__half *>(presplit);
    switch (P) {
    case 4: k_blk_presplit<4><<<grid, 256, 0, s>>>(L, begin, end, M, A, pscale); break;
    case 6: k_blk_presplit<6><<<grid, 256, 0, s>>>(L, begin, end, M, A, pscale); break;
    case 8: k_blk_presplit<8><<<grid, 256, 0, s>>>(L, begin, end, M, A, pscale); break;
    case 10: k_blk_presplit<10><<<grid, 256, 0, s>>>(L, begin, end, M, A, pscale); break;
    }
    note_launches(1);
}

template <int P>
static int launch_blk_t(int L, const int32_t *begin, const int32_t *end, const void *presplit,
                        const int8_t *pscale, const void *table, float *Lc, float *Lpart, int *status, cudaStream_t s,
                        int max_ctas)
{
    using C = BlkCfg<P>;
    constexpr CUtensorMapSwizzle kSw = CU_TENSOR_MAP_SWIZZLE_64B;
    PFN_cuTensorMapEncodeTiled_v12000 enc = tmap_encoder();
    if (!enc) return -1;
    BlkParams prm;  // the kernel parameter (copied at launch)
    memset(&prm, 0, sizeof(prm));
    prm.L = L;
    const cuuint64_t KD = C::KD, KW = C::KW;
    const int *gexp = reinterpret_cast<const int *>(static_cast<const __half *>(table) + 26 * 2 * KD * KW);
    int ntiles = 0;
    for (int l = 2; l <= L; ++l) {
        const int pg = 1 << (l - 1);
        const int bx = pg < 8 ? pg : 8, by = pg < 4 ? pg : 4, bz = by;
        prm.tile_lo[l] = ntiles;
        ntiles += (pg / bx) * (pg / by) * (pg / bz) * C::NTILES;
        void *A = const_cast<__half *>(static_cast<const __half *>(presplit) + (size_t)blk_parents_before(l - 1) * 2 * KW);
        const cuuint64_t dims[5] = {KW, 2, (cuuint64_t)pg, (cuuint64_t)pg, (cuuint64_t)pg};
        const cuuint64_t strides[4] = {KW * 2, KW * 4, KW * 4 * pg, KW * 4 * pg * pg};
        const cuuint32_t box[5] = {(cuuint32_t)kBlkCh, 1, (cuuint32_t)bx, (cuuint32_t)by, (cuuint32_t)bz};
        const cuuint32_t es[5] = {1, 1, 1, 1, 1};
        if (enc(&prm.tmA[l], CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 5, A, dims, strides, box, es,
                CU_TENSOR_MAP_INTERLEAVE_NONE, kSw, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
            return -1;
    }
    prm.tile_lo[L + 1] = ntiles;
    prm.ksplit = m2l_blk_ksplit(P, L);
    prm.part_stride = level_offset(L + 1) * C::PP;
    if (prm.ksplit > 1 && !Lpart) return -1;
    {
        const cuuint64_t dims[4] = {KW, KD, 2, 26};
        const cuuint64_t strides[3] = {KW * 2, KD * KW * 2, KD * KW * 4};
        const cuuint32_t box[4] = {(cuuint32_t)kBlkCh, (cuuint32_t)C::NT, 1, 1};
        const cuuint32_t es[4] = {1, 1, 1, 1};
        if (enc(&prm.tmB, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 4, const_cast<void *>(table), dims, strides, box, es,
                CU_TENSOR_MAP_INTERLEAVE_NONE, kSw, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
            return -1;
    }
    auto kern = k_m2l_blk<P>;
    cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)C::kSmemBytes);
    const int nctas = ntiles * prm.ksplit;
    const int step = max_ctas > 0 ? max_ctas : nctas;
    for (int t0 = 0; t0 < nctas; t0 += step) {
        prm.tile0 = t0;
        const int gsz = nctas - t0 < step ? nctas - t0 : step;
        kern<<<gsz, kBlkThreads, C::kSmemBytes, s>>>(prm, begin, end, pscale, gexp, Lc, Lpart, status);
        note_launches(1);
    }
    const int64_t npar = blk_parents_before(L), PP4 = C::PP / 4;
    k_blk_finish<P><<<(unsigned)((npar * PP4 + 31) / 32), 256, 0, s>>>(
        (int)npar, prm.ksplit, prm.part_stride / 4, begin, end,
        reinterpret_cast<const float4 *>(prm.ksplit > 1 ? Lpart : Lc), reinterpret_cast<float4 *>(Lc));
    note_launches(1);
    return 0;
}

// M2L of levels 2..L of the uniform tree (table: launch_build_m2l_blk; presplit/pscale:
// launch_blk_presplit after the upward pass); -1 if the tensor maps cannot be encoded
int launch_m2l_blk(int P, int L, const int32_t *begin, const int32_t *end, const void *presplit,
                   const int8_t *pscale, const void *table, float *Lc, float *Lpart, int *status, cudaStream_t s,
                   int max_ctas)
{
    if (L < 2) return 0;
    switch (P) {
    case 4: return launch_blk_t<4>(L, begin, end, presplit, pscale, table, Lc, Lpart, status, s, max_ctas);
    case 6: return launch_blk_t<6>(L, begin, end, presplit, pscale, table, Lc, Lpart, status, s, max_ctas);
    case 8: return launch_blk_t<8>(L, begin, end, presplit, pscale, table, Lc, Lpart, status, s, max_ctas);
    case 10: return launch_blk_t<10>(L, begin, end, presplit, pscale, table, Lc, Lpart, status, s, max_ctas);
    }
    return -1;
}

// ---- adaptive tree ----------------------------------------------------------------------------
size_t m2l_ablk_presplit_bytes(int P, int64_t ucap) { return (size_t)(ucap + 1) * 2 * blk_kw(P) * sizeof(__half); }

int64_t m2l_ablk_tiles_units(int64_t ucap) { return (ucap + kBlkRows - 1) / kBlkRows * kBlkRows; }

size_t m2l_ablk_src_bytes(int64_t ucap) { return (size_t)m2l_ablk_tiles_units(ucap) * 26 * sizeof(int32_t); }

// offset ranges per tile from the particle count and leaf size alone (an estimate of the units:
// half of n / leaf_size, as on Plummer spheres; 400,009 particles, leaf 64: 3,077), so that
// evaluations of the same count split alike whatever their trees (a captured batch and the same
// instance alone sum in the same order)
int m2l_ablk_ksplit(int P, int64_t n, int leaf_size)
{
    const int nt = P == 4 ? BlkCfg<4>::NTILES : P == 6 ? BlkCfg<6>::NTILES
                 : P == 8 ? BlkCfg<8>::NTILES : BlkCfg<10>::NTILES;
    const int64_t units = n / (2 * (int64_t)(leaf_size > 0 ? leaf_size : 1)) + 1;
    return blk_ranges((units + kBlkRows - 1) / kBlkRows * nt);
}

void launch_ablk_prep(int P, Span cells, int64_t ucap, const int32_t *level, const int32_t *nchild,
                      const int32_t *child_of, const int32_t *coll, const float *M, uint32_t *flag, uint32_t *scan,
                      uint32_t *scan_tmp, int32_t *unit_of, int32_t *units, int32_t *n_units, void *Apre,
                      int8_t *uscale, int32_t *src, cudaStream_t s)
{
    const unsigned gc = (unsigned)((cells.cap + 255) / 256);
    k_ablk_flags<<<gc, 256, 0, s>>>(cells, level, nchild, flag);
    launch_exclusive_scan(flag, scan, cells.cap, scan_tmp, s);
    k_ablk_units<<<gc, 256, 0, s>>>(cells, flag, scan, unit_of, units, n_units);
    const int64_t zrow = ucap;
    const unsigned gp = (unsigned)((ucap + 1 + 7) / 8);
    __half *A = static_cast<__half *>(Apre);
    switch (P) {
    case 4: k_ablk_presplit<4><<<gp, 256, 0, s>>>(n_units, zrow, units, child_of, M, A, uscale); break;
    case 6: k_ablk_presplit<6><<<gp, 256, 0, s>>>(n_units, zrow, units, child_of, M, A, uscale); break;
    case 8: k_ablk_presplit<8><<<gp, 256, 0, s>>>(n_units, zrow, units, child_of, M, A, uscale); break;
    case 10: k_ablk_presplit<10><<<gp, 256, 0, s>>>(n_units, zrow, units, child_of, M, A, uscale); break;
    }
    const int64_t up = m2l_ablk_tiles_units(ucap);
    k_ablk_src<<<(unsigned)((up * 26 + 255) / 256), 256, 0, s>>>(n_units, up, zrow, units, coll, unit_of, src);
    note_launches(4);
}

// How the units share V: `chunk` units at a time, the first `split` of them with their ranges apart (whole
// tiles).  Captured evaluations (uexp < ucap) size V by a quarter more than the units expected, and
// the others take their ranges in turn in the same launch; where there is one range, half the units
// at a time (four sets of 1,000,000 particles, p = 10: 4.4 GB -> 3.7, 10.98 ms -> 11.02; chunks of the
// expected units 2.9 GB and 11.18 ms).  A chunk's classes fit 1 GB: a tree of more units (at p = 10
// 335,000, of about 20M Plummer particles) takes its tiles in turns instead of 3.2 KB a unit.
struct AblkUnits {
    int64_t chunk, split;
    AblkUnits(int P, int64_t ucap, int64_t uexp, int ksplit)
    {
        const int64_t all = m2l_ablk_tiles_units(ucap), most = (int64_t(1) << 30) / ((int64_t)ksplit * 32 * P * P);
        split = std::min(all, m2l_ablk_tiles_units(std::max<int64_t>(1, uexp + uexp / 4)));
        if (ksplit > 1 && split < all)
            chunk = all;
        else
            split = chunk = std::min(std::max(split, m2l_ablk_tiles_units(all / 2)),
                                     std::max<int64_t>(kBlkRows, most / kBlkRows * kBlkRows));
    }
};

template <int P>
static int launch_ablk_t(int64_t ucap, int64_t uexp, const int32_t *n_units, const int32_t *units, const int32_t *child_of,
                         const int32_t *src, const void *Apre, const int8_t *uscale, const void *table, float *Lc,
                         float *V, int ksplit, int *status, cudaStream_t s, int max_ctas)
{
    using C = BlkCfg<P>;
    constexpr CUtensorMapSwizzle kSw = CU_TENSOR_MAP_SWIZZLE_64B;
    PFN_cuTensorMapEncodeTiled_v12000 enc = tmap_encoder();
    if (!enc) return -1;
    AblkParams prm;
    memset(&prm, 0, sizeof(prm));
    const cuuint64_t KD = C::KD, KW = C::KW;
    const int *gexp = reinterpret_cast<const int *>(static_cast<const __half *>(table) + 26 * 2 * KD * KW);
    {
        const cuuint64_t dims[4] = {KW, KD, 2, 26};
        const cuuint64_t strides[3] = {KW * 2, KD * KW * 2, KD * KW * 4};
        const cuuint32_t box[4] = {(cuuint32_t)kBlkCh, (cuuint32_t)C::NT, 1, 1};
        const cuuint32_t es[4] = {1, 1, 1, 1};
        if (enc(&prm.tmB, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 4, const_cast<void *>(table), dims, strides, box, es,
                CU_TENSOR_MAP_INTERLEAVE_NONE, kSw, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
            return -1;
    }
    prm.ksplit = ksplit;
    prm.zrow = ucap;
    const AblkUnits lay(P, ucap, uexp, ksplit);
    const bool seq = lay.split < lay.chunk;
    auto kern = seq ? k_m2l_ablk<P, true> : k_m2l_ablk<P, false>;
    auto finish = seq ? k_ablk_finish<P, true> : k_ablk_finish<P, false>;
    cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)C::kSmemBytes);
    for (int64_t u0 = 0; u0 < ucap; u0 += lay.chunk) {
        const int64_t n = std::min(lay.chunk, ucap - u0), n_split = std::min(lay.split, n);
        prm.ut0 = u0 / kBlkRows;
        prm.part_stride = n_split * C::KD;
        prm.seq0 = (int)((n_split + kBlkRows - 1) / kBlkRows * C::NTILES * ksplit);
        const int nctas = prm.seq0 + (int)((n - n_split + kBlkRows - 1) / kBlkRows * C::NTILES);
        const int step = max_ctas > 0 ? max_ctas : nctas;
        for (int t0 = 0; t0 < nctas; t0 += step) {
            prm.tile0 = t0;
            const int gsz = nctas - t0 < step ? nctas - t0 : step;
            kern<<<gsz, kAblkThreads, C::kSmemBytes, s>>>(prm, n_units, src, static_cast<const __half *>(Apre), uscale,
                                                          gexp, V, status);
            note_launches(1);
        }
        finish<<<(unsigned)((n * (C::PP / 4) + 31) / 32), 256, 0, s>>>(
            n_units, u0, (uint32_t)n, (uint32_t)n_split, ksplit, prm.part_stride / 4, units, child_of,
            reinterpret_cast<const float4 *>(V), reinterpret_cast<float4 *>(Lc));
        note_launches(1);
    }
    return 0;
}

size_t m2l_ablk_class_bytes(int P, int64_t ucap, int64_t uexp, int ksplit)
{
    const AblkUnits lay(P, ucap, uexp, ksplit);
    const int64_t n = std::min(lay.chunk, ucap);
    return (size_t)((ksplit - 1) * std::min(lay.split, n) + n) * 8 * P * P * sizeof(float);
}

int launch_m2l_ablk(int P, int64_t ucap, int64_t uexp, const int32_t *n_units, const int32_t *units, const int32_t *child_of,
                    const int32_t *src, const void *Apre, const int8_t *uscale, const void *table, float *Lc,
                    float *V, int ksplit, int *status, cudaStream_t s, int max_ctas)
{
    if (ucap <= 0) return 0;
    switch (P) {
    case 4: return launch_ablk_t<4>(ucap, uexp, n_units, units, child_of, src, Apre, uscale, table, Lc, V, ksplit, status, s, max_ctas);
    case 6: return launch_ablk_t<6>(ucap, uexp, n_units, units, child_of, src, Apre, uscale, table, Lc, V, ksplit, status, s, max_ctas);
    case 8: return launch_ablk_t<8>(ucap, uexp, n_units, units, child_of, src, Apre, uscale, table, Lc, V, ksplit, status, s, max_ctas);
    case 10: return launch_ablk_t<10>(ucap, uexp, n_units, units, child_of, src, Apre, uscale, table, Lc, V, ksplit, status, s, max_ctas);
    }
    return -1;
}

}  // namespace gbfmm

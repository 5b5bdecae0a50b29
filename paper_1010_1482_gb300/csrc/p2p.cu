// P2P near field (Section "The P2P kernel implementation", Listings 1-2) and the direct
// all-pairs sum (Eq. 1), FP32 with the reciprocal square root.
//
// Pair rule (both kernels): with d = x_i - x_j and d2 = |d|^2,
//   phi_i  += q_j / sqrt(d2 + eps2),   grad_i -= q_j d / (d2 + eps2)^(3/2),
// and pairs with d2 == 0 (the particle itself, exact duplicates) contribute nothing.
//
// Decomposition (k_p2p_ws): one producer warp and four consumer warps per CTA; a CTA takes
// every gridDim.x-th target leaf.  The producer finds a leaf's neighbour rows (the uniform tree's
// <= 27 cells by their grid position, or an adaptive leaf's U list), puts the leaf's own cell first, and copies the rows'
// particles with 1D bulk copies into one of two shared-memory stages while the consumers work on
// the other.  Each consumer thread holds two targets; when the leaf has fewer target slots than
// there are consumers the threads form G groups that split the sources round-robin, so the lanes
// stay busy for leaves of any occupancy (the paper instead pads targets to the block size).  Each
// thread sums its share in FP32; the group partials are combined per target with compensated
// (Kahan) summation.  Then either the far-field value is added the same way and the result
// written to the caller's original particle order, or (FMM) the compensated sums are stored for
// L2P, which adds the far field and writes the output.
#include "common.cuh"
#include "ptx.cuh"

#include <cooperative_groups.h>

#include <algorithm>

namespace gbfmm {

// The pair rule for two targets at once, in packed FP32 (fma.rn.f32x2 and its kin: two lanes per
// instruction), against one source; the zero-distance test only where MASK (the targets' own cell).
// nx, ny, nz: the targets' negated coordinates; gx, gy, gz: the gradient's sums.  The loop
// of scalar pairs was bound by instruction issue: of its own, 2.02e12 pairs/s scalar, 2.24e12 packed.
template <bool SOFT, bool MASK>
GB_DEV void pair2(uint64_t nx, uint64_t ny, uint64_t nz, float4 s, uint64_t eps2, uint64_t &phi, uint64_t &gx,
                  uint64_t &gy, uint64_t &gz)
{
    const uint64_t dx = add2(pack2(s.x, s.x), nx), dy = add2(pack2(s.y, s.y), ny), dz = add2(pack2(s.z, s.z), nz);
    const uint64_t d2 = fma2(dx, dx, fma2(dy, dy, mul2(dz, dz)));
    float a, b;
    unpack2(SOFT ? add2(d2, eps2) : d2, a, b);
    float ia = rsqrt_ftz(a), ib = rsqrt_ftz(b);
    if (MASK) {
        if (SOFT) unpack2(d2, a, b);
        ia = a > 0.f ? ia : 0.f;
        ib = b > 0.f ? ib : 0.f;
    }
    const uint64_t inv = pack2(ia, ib), w = mul2(pack2(s.w, s.w), inv);
    phi = add2(phi, w);
    const uint64_t w3 = mul2(mul2(w, inv), inv);
    gx = fma2(dx, w3, gx);
    gy = fma2(dy, w3, gy);
    gz = fma2(dz, w3, gz);
}

// ---- warp-specialised P2P: one producer warp stages, four consumer warps apply the pair rule ---
//
// A CTA takes the leaves blockIdx.x, blockIdx.x + gridDim.x, ...  The producer warp finds a
// leaf's neighbour rows (lane e holds row e of a block of up to 32: its first particle and count):
// on the uniform tree (UNI) from the cells' Morton positions, one leaf ahead, so that a leaf costs
// one round of loads and no list is built (two list kernels and a scan less: an evaluation of 4,096
// particles 114 -> 91 us, of 5,000,000 3157 -> 3046); on the adaptive tree from the leaf's U list.  It
// moves the target's own cell to the front of its block (only its sources pay for the
// zero-distance test), scans the counts across the warp, and copies the rows' particles
// (contiguous float4 runs of the sorted array) with 1D bulk copies into one of two stage buffers
// of kP2PCap sources; the stage's full barrier completes when the bytes have landed.  The
// consumers apply the pair rule to a stage while the producer fills the other, so a leaf's list
// reads, row copies and the previous leaf's reduction overlap the pair loop.  Targets: 2 per
// consumer thread; when a leaf has fewer target slots than there are consumers the threads form G
// groups that take the staged sources round-robin; group partials are combined with compensated
// sums, in group order, a thread per target and component.  Small uniform trees, whose leaves are
// fewer than the CTAs that fit, give a leaf's targets to `parts` CTAs.  Every wait is bounded: on expiry the kernel raises kStatusTimeout,
// stops, and returns once its own copies have landed (bounded again).
// Bound by the FP32 pipe and its issue (13 operations and a MUFU per pair).  Alone, scalar pairs and
// a one-warp reduction -> packed pairs, the reduction over all threads and stages of equal size:
// 1M particles (mean 32 per leaf) 522 -> 493 us, 5M (19 per leaf) 1852 -> 1648, 400,009 Plummer
// 222 -> 190; 16M Plummer step 26.76 -> 25.61 ms.
// Sources per stage: the most that leaves room for 8 CTAs per SM (5M uniform, 19 per leaf, about 515
// sources a leaf: 512 a stage gave half the leaves a second stage, step 2705 -> 2672 us; 1M 1002 -> 993).
// The loop unrolled by 4: by 3, 2, 8 the 1M step took 1146, 1155, 1107 us; 9 CTAs of 40 registers were
// faster at 1M (986) and slower at 5M (2753), 6 of 64 slower (1131, 3204), as were 96 or 192 consumers.
constexpr int kP2PCap = 576;
constexpr int kP2PConsumers = 128;
constexpr int kP2PWsThreads = kP2PConsumers + 32;
constexpr int kP2PTargets = 2 * kP2PConsumers;  // targets per pass over the sources

struct P2PItem {
    int b0;     // the leaf's first particle (sorted order); -1 ends the stream
    int T;      // one past the last target this CTA takes
    int tc;     // first target of this pass
    int chunk;  // sources staged (0: none, the pass only ends)
    int mend;   // leading staged sources of the target's own cell (zero-distance test)
    int flags;  // 1: first stage of the pass, 2: last stage of the pass, 4: targets are staged at tc
};

template <bool SOFT, bool UNI>
__global__ void __launch_bounds__(kP2PWsThreads, 8) k_p2p_ws(int L, const int32_t *__restrict__ leaves, Span lv,
                                                           int64_t nleaf, int parts, const float4 *__restrict__ sx,
                                                           const int32_t *__restrict__ begin,
                                                           const int32_t *__restrict__ end,
                                                           const uint32_t *__restrict__ p2p_offs,
                                                           const int32_t *__restrict__ p2p_ids,
                                                           const float4 *__restrict__ far,
                                                           const uint32_t *__restrict__ perm, float eps2,
                                                           float4 *__restrict__ out, float4 *__restrict__ near,
                                                           int *status)
{
    // two stages: the consumers read one while the producer's copies fill the other
    __shared__ __align__(128) float4 buf[2][kP2PCap];
    __shared__ float4 red[2][2][kP2PConsumers];
    __shared__ P2PItem item[2];
    __shared__ __align__(8) uint64_t full[2], empty[2], redbar[2];
    __shared__ volatile int abort_flag;
    const int tid = threadIdx.x, lane = tid & 31;
    if (tid == 0) {
        for (int k = 0; k < 2; ++k) {
            mbar_init(&full[k], 1);
            mbar_init(&empty[k], kP2PConsumers / 32);
            mbar_init(&redbar[k], kP2PConsumers);
        }
        abort_flag = 0;
        fence_mbar_init();
    }
    __syncthreads();
    const int64_t count = UNI ? nleaf * parts : span_count(lv);  // UNI: item li = part li % parts of leaf li / parts

    if (tid >= kP2PConsumers) {  // ---------------- producer warp
        int stage = 0;
        uint32_t used = 0u, par = 0u;  // per stage: filled before; parity of its last fill
        bool ok = true;
        // claim the stage: wait until the consumers have released its previous fill
        auto claim = [&]() -> bool {
            if (((used >> stage) & 1u) &&
                !mbar_wait_bounded(&empty[stage], (par >> stage) & 1u, kWaitLimitNs, &abort_flag)) {
                abort_flag = 1;
                if (status) atomicOr(status, kStatusTimeout);
            }
            return !abort_flag;
        };
        auto advance = [&] {
            par = ((used >> stage) & 1u) ? par ^ (1u << stage) : par;
            used |= 1u << stage;
            stage ^= 1;
        };
        // publish one stage (lane 0); a stage with no sources completes on the arrival alone
        auto publish = [&](const P2PItem &v) {
            if (lane == 0) {
                item[stage] = v;
                if (v.chunk > 0)
                    mbar_expect_tx(&full[stage], (uint32_t)v.chunk * 16u);
                else
                    mbar_arrive(&full[stage]);
            }
            __syncwarp();
        };
        // the uniform tree's rows, by position: lane e holds the neighbour at offset code e (13: the
        // leaf itself); cells outside the grid and empty cells count 0
        auto grid_row = [&](int64_t li, int &cb, int &cn) {
            cb = cn = 0;
            if (li >= count || lane >= 27) return;
            int x, y, z;
            demorton3((uint32_t)(li / parts), x, y, z);
            x += lane % 3 - 1;
            y += (lane / 3) % 3 - 1;
            z += lane / 9 - 1;
            const int side = 1 << L;
            if (x < 0 || y < 0 || z < 0 || x >= side || y >= side || z >= side) return;
            const int64_t c = level_offset(L) + morton3((uint32_t)x, (uint32_t)y, (uint32_t)z);
            cb = begin[c];
            cn = end[c] - cb;
        };
        int nb = 0, nn = 0;  // the next leaf's rows, loaded while the current one is staged
        if (UNI) grid_row(blockIdx.x, nb, nn);
        for (int64_t li = blockIdx.x; ok && li < count; li += gridDim.x) {
            const int gb = nb, gn = nn;
            int b0, T, nrow, t0 = 0, t1;  // targets [t0, t1) of the leaf's T particles
            uint32_t r0 = 0;
            if (UNI) {
                grid_row(li + gridDim.x, nb, nn);
                b0 = __shfl_sync(~0u, gb, 13);
                T = __shfl_sync(~0u, gn, 13);
                const int per = (T + parts - 1) / parts;
                t0 = (int)(li % parts) * per;
                t1 = min(T, t0 + per);
                if (t0 >= t1) continue;
                nrow = 27;
            } else {
                const int64_t g = leaves[li];
                b0 = begin[g];
                T = end[g] - b0;
                if (T <= 0) continue;
                t1 = T;
                r0 = p2p_offs[g];
                nrow = (int)(p2p_offs[g + 1] - r0);
            }
            for (int tc = t0; ok && tc < t1; tc += kP2PTargets) {
                const int Tc = min(t1 - tc, kP2PTargets);
                bool emitted = false;
                for (int rb = 0; ok && rb < nrow; rb += 32) {
                    const int nr = min(32, nrow - rb);
                    const bool last_rb = rb + 32 >= nrow;
                    int cb = 0, cn = 0;
                    if (UNI) {
                        cb = gb;
                        cn = gn;
                    } else if (lane < nr) {
                        const int c = p2p_ids[r0 + rb + lane];
                        cb = begin[c];
                        cn = end[c] - cb;
                    }
                    // the target's own cell first
                    const unsigned self = __ballot_sync(~0u, lane < nr && cb == b0 && cn == T);
                    const int k = self ? __ffs(self) - 1 : 0;
                    const int cb0 = __shfl_sync(~0u, cb, 0), cn0 = __shfl_sync(~0u, cn, 0);
                    const int cbk = __shfl_sync(~0u, cb, k), cnk = __shfl_sync(~0u, cn, k);
                    if (self && k > 0) {
                        if (lane == 0) cb = cbk, cn = cnk;
                        else if (lane == k) cb = cb0, cn = cn0;
                    }
                    int incl = cn;
#pragma unroll
                    for (int d = 1; d < 32; d <<= 1) {
                        const int v = __shfl_up_sync(~0u, incl, d);
                        if (lane >= d) incl += v;
                    }
                    const int pref = incl - cn, S = __shfl_sync(~0u, incl, 31);
                    const int nself = self ? T : 0;
                    const int per_stage = S > 0 ? (S + (S + kP2PCap - 1) / kP2PCap - 1) / ((S + kP2PCap - 1) / kP2PCap) : 1;
                    for (int sc = 0; sc < S; sc += per_stage) {  // stages of about equal size
                        const int chunk = min(per_stage, S - sc);
                        if (!claim()) {
                            ok = false;
                            break;
                        }
                        const bool last = last_rb && sc + chunk >= S;
                        const bool staged = rb == 0 && sc == 0 && nself > 0 && tc + Tc <= chunk;
                        publish(P2PItem{b0, t1, tc, chunk, max(0, min(chunk, nself - sc)),
                                        (emitted ? 0 : 1) | (last ? 2 : 0) | (staged ? 4 : 0)});
                        const int lo = max(pref, sc), hi = min(pref + cn, sc + chunk);
                        if (hi > lo)
                            tma_bulk_g2s(&buf[stage][lo - sc], &sx[cb + (lo - pref)], (uint32_t)(hi - lo) * 16u,
                                         &full[stage]);
                        emitted = true;
                        advance();
                    }
                    if (ok && last_rb && S == 0) {  // the pass ends on an empty block
                        if (!claim()) {
                            ok = false;
                            break;
                        }
                        publish(P2PItem{b0, t1, tc, 0, 0, (emitted ? 0 : 1) | 2});
                        emitted = true;
                        advance();
                    }
                }
                if (ok && !emitted) {  // no neighbour rows at all
                    if (!claim()) {
                        ok = false;
                        break;
                    }
                    publish(P2PItem{b0, t1, tc, 0, 0, 3});
                    advance();
                }
            }
        }
        if (ok && claim()) {  // end of stream
            publish(P2PItem{-1, 0, 0, 0, 0, 0});
            advance();
        }
        if (abort_flag) {
            // stopped early: return only once this warp's copies have landed
            for (int k = 0; k < 2; ++k)
                if ((used >> k) & 1u) mbar_wait_bounded(&full[k], ((par >> k) & 1u), kWaitLimitNs, nullptr);
        }
        return;
    }

    // -------------------------------------------------- consumer warps
    int stage = 0, rpar = 0;
    uint32_t fpar = 0u, rphase = 0u;  // per stage / per reduction buffer: parity of the next phase
    int slots = 1, G = 1, slot = 0, grp = 0, Tc = 0;
    // two targets per thread, packed: negated coordinates, sums
    uint64_t nx = 0, ny = 0, nz = 0, phi = 0, gx = 0, gy = 0, gz = 0;
    const uint64_t e2 = pack2(eps2, eps2);
    while (true) {
        if (!mbar_wait_bounded(&full[stage], (fpar >> stage) & 1u, kWaitLimitNs, &abort_flag) || abort_flag) {
            if (!abort_flag) {
                abort_flag = 1;
                if (status) atomicOr(status, kStatusTimeout);
            }
            return;
        }
        const P2PItem it = item[stage];
        if (it.b0 < 0) return;
        const float4 *src = buf[stage];
        if (it.flags & 1) {  // a new pass: its targets
            Tc = min(it.T - it.tc, kP2PTargets);
            slots = (Tc + 1) / 2;
            G = kP2PConsumers / slots;
            slot = tid % slots;
            grp = tid / slots;
            // a missing target repeats the slot's first one; its result is discarded
            const int ta = 2 * slot, tb = ta + 1 < Tc ? ta + 1 : ta;
            const float4 A = (it.flags & 4) ? src[it.tc + ta] : __ldg(&sx[it.b0 + it.tc + ta]);
            const float4 B = (it.flags & 4) ? src[it.tc + tb] : __ldg(&sx[it.b0 + it.tc + tb]);
            nx = pack2(-A.x, -B.x), ny = pack2(-A.y, -B.y), nz = pack2(-A.z, -B.z);
            phi = gx = gy = gz = 0;
        }
        if (grp < G) {
            int j = grp;
            for (; j < it.mend; j += G) pair2<SOFT, true>(nx, ny, nz, src[j], e2, phi, gx, gy, gz);
#pragma unroll 4
            for (; j < it.chunk; j += G) pair2<SOFT, false>(nx, ny, nz, src[j], e2, phi, gx, gy, gz);
        }
        __syncwarp();
        if (lane == 0) mbar_arrive(&empty[stage]);
        fpar ^= 1u << stage;
        stage ^= 1;
        if (!(it.flags & 2)) continue;
        // end of the pass: combine the groups' partials per target.  red alternates between two
        // buffers, and every consumer waits for the pass's arrivals, so a pass's writes never
        // meet the previous pass's reads.
        {
            float4 va, vb;
            unpack2(phi, va.x, vb.x);
            unpack2(gx, va.y, vb.y);
            unpack2(gy, va.z, vb.z);
            unpack2(gz, va.w, vb.w);
            red[rpar][0][tid] = va;
            red[rpar][1][tid] = vb;
        }
        mbar_arrive(&redbar[rpar]);
        if (!mbar_wait_bounded(&redbar[rpar], (rphase >> rpar) & 1u, kWaitLimitNs, &abort_flag)) {
            if (!abort_flag) {
                abort_flag = 1;
                if (status) atomicOr(status, kStatusTimeout);
            }
            return;
        }
        rphase ^= 1u << rpar;
        // one component of one target per thread (e: target parity, slot, component)
        for (int e = tid; e < 8 * slots; e += kP2PConsumers) {
            const int cp = e & 3, hs = e >> 2, h = hs >= slots, sl = hs - (h ? slots : 0), t = 2 * sl + h;
            if (t >= Tc) continue;
            const int64_t i = it.b0 + it.tc + t;
            const float *r = reinterpret_cast<const float *>(&red[rpar][h][sl]) + cp;
            Kahan a{0.f, 0.f};
            for (int k = 0; k < G; ++k) a.add(r[4 * k * slots]);
            if (near) {  // the compensated sums so far; the far field is added by L2P
                float *nr = reinterpret_cast<float *>(near + 2 * i) + cp;
                nr[0] = a.s;
                nr[4] = a.c;
                continue;
            }
            if (far) a.add(reinterpret_cast<const float *>(far + i)[cp]);
            reinterpret_cast<float *>(out + perm[i])[cp] = a.s;
        }
        rpar ^= 1;
    }
}

// ---- launchers --------------------------------------------------------------------------------
// CTAs resident per SM, and the largest shared-memory carveout so that the kernel's CTAs can
// share an SM with the far field's when both run at once
static int p2p_blocks_per_sm()
{
    static const int b = [] {
        for (auto k : {k_p2p_ws<false, false>, k_p2p_ws<false, true>, k_p2p_ws<true, false>, k_p2p_ws<true, true>})
            cudaFuncSetAttribute(k, cudaFuncAttributePreferredSharedMemoryCarveout,
                                 (int)cudaSharedmemCarveoutMaxShared);
        int v = 0;
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&v, k_p2p_ws<false, false>, kP2PWsThreads, 0);
        return v > 0 ? v : 1;
    }();
    return b;
}

// nleaf: the leaves (uniform tree) or the capacity of the listed leaves (lv.cap).  Each CTA takes
// about kP2PLeavesPerCta of them (never fewer CTAs than fit on the GPU at once): enough leaves
// that the producer's staging of one hides behind the pair loop of another, few enough that CTAs
// retire often and the far field's kernels, beside P2P on the other stream, get SMs.  Measured on
// the 1M uniform step (p = 10): 1, 2, 4, 8 leaves and one persistent wave gave P2P 0.528, 0.520,
// 0.525, 0.541, 0.596 ms alone and 1.158, 1.152, 1.163, 1.189, 1.248 ms for the forked step; on
// 16M Plummer (p = 8) P2P took 8.91, 7.97, 9.29 ms with 1, 4 and one wave.
constexpr int kP2PLeavesPerCta = 4;
constexpr int kP2PMaxParts = 16, kP2PWave = kSms * 8;
// the evaluating context's choice (gbfmm_set_p2p_leaves_per_cta, gbfmm_tune), set on entry to an
// evaluation by the thread that issues its launches; 0: kP2PLeavesPerCta
static thread_local int tl_leaves_per_cta = 0;
void set_p2p_leaves_per_cta(int leaves) { tl_leaves_per_cta = leaves; }

static void launch_leaf(int64_t nleaf, int L, const int32_t *leaves, const float4 *sx, const int32_t *begin,
                        const int32_t *end, const uint32_t *offs, const int32_t *ids, const float4 *far,
                        const uint32_t *perm, float eps2, float4 *out, float4 *near, int *status, cudaStream_t s,
                        Span lv = Span{})
{
    const int64_t resident = (int64_t)sm_count() * p2p_blocks_per_sm();
    // small uniform trees: a leaf's targets over up to kP2PMaxParts CTAs, so that the launch has one
    // wave of CTAs (4,096 particles, 64 leaves: 39 -> 10.5 us, packed pairs included).  Fixed by the depth: the sums do not depend on
    // the launch shape.
    const int parts = leaves ? 1 : (int)std::max<int64_t>(1, std::min<int64_t>(kP2PMaxParts, kP2PWave / nleaf));
    const int lpc = tl_leaves_per_cta > 0 ? tl_leaves_per_cta : kP2PLeavesPerCta;
    int64_t grid = (nleaf + lpc - 1) / lpc;
    grid = std::min<int64_t>(nleaf * parts, std::max<int64_t>(grid, resident));
    const bool soft = eps2 > 0.f;
    auto k = leaves ? (soft ? k_p2p_ws<true, false> : k_p2p_ws<false, false>)
                    : (soft ? k_p2p_ws<true, true> : k_p2p_ws<false, true>);
    k<<<(unsigned)grid, kP2PWsThreads, 0, s>>>(L, leaves, lv, nleaf, parts, sx, begin, end, offs, ids, far, perm, eps2, out,
                                               near, status);
    note_launches(1);
}

void launch_p2p(int L, int64_t n, const float4 *sx, const int32_t *begin, const int32_t *end, const float4 *far,
                const uint32_t *perm, float eps2, float4 *out, int *status, cudaStream_t s)
{
    if (n <= 0) return;
    launch_leaf(int64_t(1) << (3 * L), L, nullptr, sx, begin, end, nullptr, nullptr, far, perm, eps2, out, nullptr,
                status, s);
}

void launch_p2p_cells(const int32_t *leaves, Span lv, int64_t n, const float4 *sx, const int32_t *begin,
                      const int32_t *end, const uint32_t *u_offs, const int32_t *u_ids, const float4 *far,
                      const uint32_t *perm, float eps2, float4 *out, int *status, cudaStream_t s)
{
    if (n <= 0 || lv.cap <= 0) return;
    launch_leaf(lv.cap, 0, leaves, sx, begin, end, u_offs, u_ids, far, perm, eps2, out, nullptr, status, s, lv);
}

void launch_p2p_near(int L, int64_t n, const float4 *sx, const int32_t *begin, const int32_t *end, float eps2,
                     float4 *near, int *status, cudaStream_t s)
{
    if (n <= 0) return;
    launch_leaf(int64_t(1) << (3 * L), L, nullptr, sx, begin, end, nullptr, nullptr, nullptr, nullptr, eps2, nullptr,
                near, status, s);
}

void launch_p2p_cells_near(const int32_t *leaves, Span lv, int64_t n, const float4 *sx, const int32_t *begin,
                           const int32_t *end, const uint32_t *u_offs, const int32_t *u_ids, float eps2, float4 *near,
                           int *status, cudaStream_t s)
{
    if (n <= 0 || lv.cap <= 0) return;
    launch_leaf(lv.cap, 0, leaves, sx, begin, end, u_offs, u_ids, nullptr, nullptr, eps2, nullptr, near, status, s, lv);
}

// Direct all-pairs sum.  A CTA takes 64 targets, two per lane in packed pairs, and its four warps
// share the sources staged in shared memory (cp.async, the next tile in flight), four sources at a
// time; a cluster of 8 CTAs splits the sources of the same targets, and the sums are added through
// distributed shared memory, warps then CTAs in order.  So a call has 8 x 4 x n_tgt / 64 warps: with
// a thread per target (256 to a CTA, every source in turn) 16,411 targets filled 65 of 152 SMs:
// 442 -> 144 us.  Bound by the FP32 pipe.
// Any two particles may coincide; the zero-distance test is made on the least of four sources' d2
// (NaN included) and only a group that fails it takes the masked rule.
//
// Targets alone fill the GPU where they are many and the sources few, and a cluster of 8 CTAs for a
// handful of sources is launches and sums only: 1,000,000 targets of 64 sources took 321 us, 256 of
// 352, 1024 of 570 (a thread per target: 39, 138, 538).  So (us, cluster of 8 / CTA alone / thread
// per target):
//   - a thread per target up to 128 sources: 64 of 1M 321 / 47 / 39, 128 of 1M 326 / 70 / 72, 64 of
//     10,000 8.2 / 6.1 / 4.2; for up to 1024 targets the cluster is as fast from 32 sources on
//     (128 of 64: 4.2 / 6.1 / 6.2);
//   - up to 1024 sources a CTA alone (SPLIT = 1) from 48 targets a source on: 256 of 10,000 8.3 / 7.2 /
//     10.3, 512 of 20,000 12.4 / 12.4 / 16.4, 1024 of 50,000 33.0 / 32.9 / 47.2, 1024 of 1M 570 / 442 / 538;
//   - else the cluster (4096 of 20,000: 45 / 64 / 102), which also keeps every sum short.
constexpr int kDirectThreads = 128, kDirectTargets = 64, kDirectTile = 512, kDirectSplit = 8;
constexpr int64_t kDirectFewSources = 128, kDirectOneSources = 1024;

// the least of four packed pairs; NaN if any of them is
GB_DEV float least8(const uint64_t (&d2)[4])
{
    float v[8], m;
#pragma unroll
    for (int u = 0; u < 4; ++u) unpack2(d2[u], v[2 * u], v[2 * u + 1]);
    asm("min.NaN.f32 %0, %1, %2, %3;" : "=f"(m) : "f"(v[0]), "f"(v[1]), "f"(v[2]));
    asm("min.NaN.f32 %0, %1, %2, %3;" : "=f"(m) : "f"(m), "f"(v[3]), "f"(v[4]));
    asm("min.NaN.f32 %0, %1, %2, %3;" : "=f"(m) : "f"(m), "f"(v[5]), "f"(v[6]));
    asm("min.NaN.f32 %0, %1, %2;" : "=f"(m) : "f"(m), "f"(v[7]));
    return m;
}

// sources S[first + step k .. + 4) of the cnt staged ones, for k = 0, 1, ...; a group cut short by cnt goes
// one source at a time
template <bool SOFT>
GB_DEV void direct_sources(const float4 *S, int cnt, int first, int step, uint64_t nx, uint64_t ny, uint64_t nz,
                           uint64_t e2, uint64_t &phi, uint64_t &gx, uint64_t &gy, uint64_t &gz)
{
    int j = first;
    for (; j + 4 <= cnt; j += step) {
        uint64_t dx[4], dy[4], dz[4], d2[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const float4 q = S[j + u];
            dx[u] = add2(pack2(q.x, q.x), nx), dy[u] = add2(pack2(q.y, q.y), ny), dz[u] = add2(pack2(q.z, q.z), nz);
            d2[u] = fma2(dx[u], dx[u], fma2(dy[u], dy[u], mul2(dz[u], dz[u])));
        }
        if (least8(d2) > 0.f) {
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const float qw = S[j + u].w;
                float a, c;
                unpack2(SOFT ? add2(d2[u], e2) : d2[u], a, c);
                const uint64_t inv = pack2(rsqrt_ftz(a), rsqrt_ftz(c)), w = mul2(pack2(qw, qw), inv);
                phi = add2(phi, w);
                const uint64_t w3 = mul2(mul2(w, inv), inv);
                gx = fma2(dx[u], w3, gx);
                gy = fma2(dy[u], w3, gy);
                gz = fma2(dz[u], w3, gz);
            }
        } else {
            for (int u = 0; u < 4; ++u) pair2<SOFT, true>(nx, ny, nz, S[j + u], e2, phi, gx, gy, gz);
        }
    }
    for (; j < cnt; ++j) pair2<SOFT, true>(nx, ny, nz, S[j], e2, phi, gx, gy, gz);
}

template <bool SOFT, int SPLIT>
__global__ void __cluster_dims__(SPLIT, 1, 1) __launch_bounds__(kDirectThreads)
    k_direct(int64_t ns, const float4 *__restrict__ src, int64_t nt, const float4 *__restrict__ tgt, float eps2,
             float4 *__restrict__ out)
{
    namespace cg = cooperative_groups;
    __shared__ __align__(16) float4 tile[2][kDirectTile];
    __shared__ float4 red[kDirectThreads / 32][kDirectTargets];
    __shared__ float4 sum[kDirectTargets];
    const cg::cluster_group cl = cg::this_cluster();
    const int rank = (int)cl.block_rank(), tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int64_t t0 = (int64_t)(blockIdx.x / SPLIT) * kDirectTargets;
    const int64_t per = (ns + SPLIT - 1) / SPLIT, s0 = rank * per, s1 = min(ns, s0 + per);
    auto target = [&](int k) { return t0 + k < nt ? __ldg(&tgt[t0 + k]) : make_float4(0.f, 0.f, 0.f, 0.f); };
    const float4 A = target(lane), B = target(lane + 32);
    const uint64_t nx = pack2(-A.x, -B.x), ny = pack2(-A.y, -B.y), nz = pack2(-A.z, -B.z), e2 = pack2(eps2, eps2);
    uint64_t phi = 0, gx = 0, gy = 0, gz = 0;
    auto stage = [&](int64_t b, int buf) {
        for (int k = tid; k < kDirectTile; k += kDirectThreads)
            if (b + k < s1) cp_async16(&tile[buf][k], &src[b + k], 16u);
        cp_async_commit();
    };
    if (s0 < s1) stage(s0, 0);
    int buf = 0;
    for (int64_t b = s0; b < s1; b += kDirectTile, buf ^= 1) {
        cp_async_wait<0>();
        __syncthreads();  // the tile is there, and the other buffer's readers are done
        if (b + kDirectTile < s1) stage(b + kDirectTile, buf ^ 1);
        const int cnt = (int)min((int64_t)kDirectTile, s1 - b);
        const float4 *S = tile[buf];
        direct_sources<SOFT>(S, cnt, 4 * warp, kDirectThreads / 8, nx, ny, nz, e2, phi, gx, gy, gz);
    }
    float4 va, vb;
    unpack2(phi, va.x, vb.x);
    unpack2(gx, va.y, vb.y);
    unpack2(gy, va.z, vb.z);
    unpack2(gz, va.w, vb.w);
    red[warp][lane] = va;
    red[warp][lane + 32] = vb;
    __syncthreads();
    auto add = [](float4 &r, const float4 &v) { r.x += v.x, r.y += v.y, r.z += v.z, r.w += v.w; };
    if (tid < kDirectTargets) {
        float4 r = red[0][tid];
#pragma unroll
        for (int w = 1; w < kDirectThreads / 32; ++w) add(r, red[w][tid]);
        sum[tid] = r;
    }
    cl.sync();
    // CTA `rank` adds the CTAs' sums of its share of the targets
    const int k = rank * (kDirectTargets / SPLIT) + tid;
    if (tid < kDirectTargets / SPLIT && t0 + k < nt) {
        float4 r = *cl.map_shared_rank(&sum[k], 0);
        for (int c = 1; c < SPLIT; ++c) add(r, *cl.map_shared_rank(&sum[k], c));
        out[t0 + k] = r;
    }
    cl.sync();  // no CTA leaves while its sums may be read
}

// Few sources: a thread per target takes every source in turn, nothing is staged twice or added up.
constexpr int kDirectFewThreads = 256;

template <bool SOFT>
__global__ void __launch_bounds__(kDirectFewThreads) k_direct_few(int ns, const float4 *__restrict__ src, int64_t nt,
                                                                  const float4 *__restrict__ tgt, float eps2,
                                                                  float4 *__restrict__ out)
{
    __shared__ float4 tile[kDirectFewSources];
    if (threadIdx.x < ns) tile[threadIdx.x] = __ldg(&src[threadIdx.x]);
    __syncthreads();
    const int64_t i = blockIdx.x * (int64_t)kDirectFewThreads + threadIdx.x;
    if (i >= nt) return;
    const float4 t = __ldg(&tgt[i]);
    float phi = 0.f, gx = 0.f, gy = 0.f, gz = 0.f;
#pragma unroll 8
    for (int j = 0; j < ns; ++j) {
        const float4 q = tile[j];
        const float dx = q.x - t.x, dy = q.y - t.y, dz = q.z - t.z;
        const float d2 = fmaf(dx, dx, fmaf(dy, dy, dz * dz));
        const float inv = d2 > 0.f ? rsqrt_ftz(SOFT ? d2 + eps2 : d2) : 0.f;
        const float w = q.w * inv, w3 = w * inv * inv;
        phi += w;
        gx = fmaf(dx, w3, gx);
        gy = fmaf(dy, w3, gy);
        gz = fmaf(dz, w3, gz);
    }
    out[i] = make_float4(phi, gx, gy, gz);
}

void launch_direct(int64_t n_src, const float4 *src, int64_t n_tgt, const float4 *tgt, float eps2, float4 *out,
                   cudaStream_t s)
{
    if (n_tgt <= 0) return;
    const bool soft = eps2 > 0.f;
    const int64_t ctas = (n_tgt + kDirectTargets - 1) / kDirectTargets;
    if (n_src <= kDirectFewSources && (n_src <= 32 || n_tgt > 1024)) {
        const unsigned grid = (unsigned)((n_tgt + kDirectFewThreads - 1) / kDirectFewThreads);
        auto k = soft ? k_direct_few<true> : k_direct_few<false>;
        k<<<grid, kDirectFewThreads, 0, s>>>((int)n_src, src, n_tgt, tgt, eps2, out);
    } else if (n_src <= kDirectOneSources && n_tgt > 48 * n_src) {
        auto k = soft ? k_direct<true, 1> : k_direct<false, 1>;
        k<<<(unsigned)ctas, kDirectThreads, 0, s>>>(n_src, src, n_tgt, tgt, eps2, out);
    } else {
        auto k = soft ? k_direct<true, kDirectSplit> : k_direct<false, kDirectSplit>;
        k<<<(unsigned)(ctas * kDirectSplit), kDirectThreads, 0, s>>>(n_src, src, n_tgt, tgt, eps2, out);
    }
    note_launches(1);
}

}  // namespace gbfmm

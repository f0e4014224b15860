// Exact DTW dynamic programming, warp-specialised: every strip of A has a
// DP warp and a cost warp, and every CTA of NS strips a reader and a writer
// warp for the border it shares with the neighbouring CTAs.  Same
// recurrence, step set, weights and tie order as the other DP kernels
// (Sec. V, Sec. II-D); only the division of labour differs.
//
//   - The strip geometry is that of the multi-row kernel: 31 R rows, lane t
//     (0..30) of the DP warp holds rows R t .. R t + R - 1 of the strip,
//     lane 31 is the ghost lane that carries the two bottom rows of the strip
//     above (cost 1e30, weight 0 on the (1,2) candidate fed the border value).
//   - The cost warp(s) of the strip compute C' = (1 - mu) - a^_i . b^_j for the
//     same rows, 8 columns (a sub-chunk) at a time (one FMA per feature, in
//     feature order, so the values are bit-identical to the other kernels'),
//     reading the frames of B from a TMA-fed ring, and hand them to the DP
//     warp through a ring of kSlots slots in shared memory.  A slot also holds
//     the strip's top border for its columns: the two bottom rows of the strip
//     above, which that strip's DP warp (or, for the first strip of a CTA, the
//     reader warp or the CTA above in its cluster) stores there.  One full
//     barrier per slot counts both, one empty barrier releases both.
//   - The DP warp runs only the recurrence: per column two shuffles, three
//     FMAs, a three-way minimum and two compares per cell.  It works one
//     sub-chunk behind its loads: in the middle of a sub-chunk it tests the
//     next slot's barrier and loads it, a load or two per column, so that
//     neither the test nor the loads (nor the queue of shared-memory accesses
//     in front of a shuffle) hold up the recurrence, and the outcome of the
//     test is looked at after the eight steps.  The strip's two bottom rows go
//     out column by column, one 8-byte store each.
//   - The last strip of a CTA hands its rows to the writer warp through a
//     ring of its own, which publishes them in global memory or, inside a
//     cluster, stores them straight into the slots of the CTA below.
//   - Every wait is bounded (DTW_ERR_TIMEOUT) and gives up when the call has
//     failed elsewhere.
#pragma once
#include "dp_device.cuh"

// The kernel templates are included by dp_split.cu (two strips per CTA) and
// dp_split4.cu (four strips per CTA), which instantiate and launch them.
namespace pardtw {
namespace {

constexpr int kGhostLane = 31;
constexpr int kOutLane = 30;    // holds the strip's two bottom rows
// Sub-chunks in flight per strip, and in the writer's ring.  In a cluster a
// slot's round trip (stored by the CTA above, released here, handed back) is
// longer than 8 sub-chunks.
template <bool kCl>
constexpr int slots_of() {
    return kCl ? 16 : 8;
}
// Uses of the slots between two CTAs of a cluster that are handed back together (20000 x
// 25000, D = 12: DP 0.996 ms with every use handed back by itself, 0.919 by 4, 0.907 by
// 8, half of the slots).
constexpr int kLinkPage = 8;
constexpr int kBorderBytes = 2 * kSub * 4;  // 8 columns of (row top-2, row top-1) pairs

// One slot holds the 8 costs of each of a lane's R rows: float4 q of lane l
// (q = 2 k + half) at [q][l], so a warp's 16-byte accesses are contiguous;
// then the top border of the 8 columns.
template <int R>
struct CostRing {
    static constexpr int kF4 = 2 * R;
    static constexpr int kBorder = kF4 * kWarp * 16;
    static constexpr int kSlotBytes = kBorder + kBorderBytes;
};

// BF16 cost: one slot holds the 8 costs of each of the 32 R rows of the
// strip row by row, kRowFloats floats per row (48-byte rows: the DP warp's
// 16-byte loads of rows 3l+k then fall in distinct bank groups), then the top
// border.
constexpr int kRowFloats = 12;
template <int R>
struct CostRingRM {
    static constexpr int kBorder = 32 * R * kRowFloats * 4;
    static constexpr int kSlotBytes = kBorder + kBorderBytes;
};
template <int R, bool kRM>
struct SlotOf {
    static constexpr int kBorder = kRM ? CostRingRM<R>::kBorder : CostRing<R>::kBorder;
    static constexpr int kBytes = kRM ? CostRingRM<R>::kSlotBytes : CostRing<R>::kSlotBytes;
};
// BF16 cost: the strip's rows of A as bf16 (32 R rows of kBfStride), and a
// ring of kBfSlots blocks of 16 frames of B (one chunk each) filled by TMA.
constexpr int kBfSlots = 4;
constexpr int kBfBlkBytes = kColsPerWord * kBfStride * 2;

// FP32 cost for D > 32 ("wide"): -a^ of the lane's R rows no longer fits in
// registers, so the strip's rows of A^ sit in shared memory (rows padded by 4
// floats: the 16-byte loads of rows 3l + k of a warp fall in distinct bank
// groups), and several cost warps share a strip, taking sub-chunks in turn
// (all 8 columns each).  So they do where one would be slower than the DP warp.
// With two strips a CTA: two (20000 x 25000 at D = 12: DP 0.907 ms, 1.056 with a third one,
// which shares the DP warp's SM sub-partition; a plan of 256 pairs 3.51 and 3.73), at
// D = 32 three (256 pairs of up to 4000 frames: 1.43 ms, 1.60 with two).  With one strip, four
// of the wide ones (24001 x 27011 at D = 100: 3.23 ms, 2.50 with six, which are not
// measured at other sizes), and three otherwise (40000 x 48000 with the BF16 cost: 2.72,
// 2.73 with four).
template <int DP, int NS, bool kBF>
struct CostCfg {
    static constexpr bool kWide = DP > 32 && !kBF;
    // cost warps a strip
    static constexpr int kNC = kWide           ? (NS == 1 ? 4 : 2)
                               : NS == 1       ? 3
                               : kBF || NS > 2 ? 1
                               : DP > 16       ? 3
                               : DP > 8        ? 2
                                               : 1;
    static constexpr int kStride = DP + 4;   // floats per row of the A tile
    // each cost warp's ring of B: frames a block, blocks
    static constexpr int kBBlk = kWide ? kColsPerWord : (DP <= 16 ? 64 : 32);
    static constexpr int kBSlots = kNC >= 2 ? 2 : 4;
};
template <int DP, int R, int NS, bool kBF, bool kCl>
struct SplitSmem {
    using Cfg = CostCfg<DP, NS, kBF>;
    // per strip slot: the cost warps' operands (B stages; A tile and B stage
    // for the BF16 cost; A tile and B stages for the wide FP32 cost), then the
    // slots
    static constexpr int kOperandBytes =
        kBF ? 32 * R * kBfStride * 2 + Cfg::kNC * kBfSlots * kBfBlkBytes
            : (Cfg::kWide ? 32 * R * Cfg::kStride * 4 : 0) +
                  Cfg::kNC * BStage<DP, Cfg::kBSlots, Cfg::kBBlk>::kWarpBytes;
    static constexpr int kStripBytes =
        kOperandBytes + slots_of<kCl>() * SlotOf<R, kBF>::kBytes;
};
// Threads of a CTA of NS strips: per strip the cost warp(s) and a DP warp,
// plus the reader and the writer.
template <int DP, int NS, bool kBF>
__host__ __device__ constexpr int split_threads() {
    return ((CostCfg<DP, NS, kBF>::kNC + 1) * NS + 2) * 32;
}

// Barrier `slot` of an array of 8-byte mbarriers, and the phase parity a
// waiter for the t-th (lifetime) use of a ring of n slots expects.
__device__ __forceinline__ unsigned bar_at(unsigned base, unsigned slot) { return base + 8 * slot; }
__device__ __forceinline__ unsigned use_parity(unsigned t, unsigned n) { return (t / n) & 1u; }

// Sub-chunks [x, y) (columns 8x .. 8y-1) that `strip` sweeps: the band's
// range of the strip, every column in the subsequence DP (a fragment's path
// may start and end anywhere), else the columns of the strip's rows that a
// path can cross (path_lo, path_hi), and the two columns before them, where
// the strip above may hold their predecessors, rounded out to whole words.
// Cells outside change nothing that a path reads, and leaving them out cuts
// the sweep of a square matrix to a third: align of 100000 x 126231 frames at
// D = 12 went from
// 24.8 to 12.2 ms, a planned batch of 256 pairs of up to 8000 frames from 11.7
// to 8.3 ms (20000 x 25000, bound by the chain of strips: 1.51 and 1.54 ms).
template <bool kAllCols = false>
__device__ __forceinline__ int2 strip_range(const DpArgs& p, int strip) {
    const int nsub = (p.Lb + kSub - 1) / kSub;
    if (kAllCols) return make_int2(0, nsub);
    if (p.ranges) return p.ranges[strip];
    const int r0 = strip * p.rps, r1 = min(r0 + p.rps, p.La) - 1;
    const int x = (max(path_lo(r0, p.La, p.Lb) - 2, 0) / kSub) & ~1;
    const int y = min(max(path_hi(r1, p.La, p.Lb), 0) / kSub + 1, nsub);
    return make_int2(x, max(y, x + 1));
}

// Where the top border of a strip's slots comes from: sub-chunks before
// link_end from the CTA above in the cluster (64 bytes of asynchronous stores
// on the full barrier), those from inf_from on have none (+inf, stored here),
// the others from another warp of the CTA (its arrival is one of the full
// barrier's two).
struct BorderSrc {
    int inf_from, link_end;
};

// The costs of sub-chunk n are in the slot (every lane has stored its own):
// arrive for them, and settle the border's share of the slot.
__device__ __forceinline__ void cost_arrive(unsigned full, unsigned border, int n,
                                            const BorderSrc& bs, int lane) {
    if (n >= bs.inf_from && lane < 2 * kSub) sts32(border + (unsigned)lane * 4u, INFINITY);
    __syncwarp();
    if (lane == 0) {
        if (n >= bs.inf_from) {
            mbar_arrive_n(full, 2);
        } else {
            if (n < bs.link_end) mbar_arrive_expect_tx(full, kBorderBytes);
            mbar_arrive(full);
        }
    }
}

// Cost warp `half` of the kNC of `strip`: every kNC-th sub-chunk of the
// sweep, in order.  Bound by the FMAs' three register operands: paired FMAs
// (two columns each, each rounded once: the values of one FMA per feature in
// feature order) take 70 cycles a column of a D = 12 strip for one warp alone
// on its SM sub-partition and 52 with two, scalar ones 64 and 60.  (A pass over
// 16 columns takes 49 and 47 but fills its slots in bursts: no faster in the
// kernel, and slower at D = 32 and where two CTAs share an SM's registers.)
template <int DP, int R, int NS, int kSlots, bool kAllCols, int kNG = DP / 4>
__device__ __forceinline__ void run_cost(const DpArgs& p, int strip, int half, int lane,
                                         unsigned cring, unsigned cfull, unsigned cempty,
                                         unsigned csub, const BorderSrc& bs,
                                         BRing<DP, CostCfg<DP, NS, false>::kBSlots,
                                               CostCfg<DP, NS, false>::kBBlk>& br) {
    using Cfg = CostCfg<DP, NS, false>;
    using S = BStage<DP, Cfg::kBSlots, Cfg::kBBlk>;
    using CR = CostRing<R>;
    constexpr int kRows = 31 * R;
    constexpr int kFG = 4;            // features per group of loads; kNG groups have some
    static_assert(S::kBlk >= kSub * Cfg::kNC, "a warp reads some of every block of B");
    const bool ghost = lane == kGhostLane;
    const int i0 = strip * kRows + lane * R;
    float na[R][DP];  // -a^_i of the lane's rows (0 in the ghost lane)
#pragma unroll
    for (int k = 0; k < R; ++k) {
        const float4* s = reinterpret_cast<const float4*>(p.Ahat + (size_t)(i0 + k) * DP);
#pragma unroll
        for (int q = 0; q < DP / 4; ++q) {
            const float4 v = ghost ? make_float4(0.f, 0.f, 0.f, 0.f) : s[q];
            na[k][4 * q] = -v.x;
            na[k][4 * q + 1] = -v.y;
            na[k][4 * q + 2] = -v.z;
            na[k][4 * q + 3] = -v.w;
        }
    }
    const float kc = ghost ? kGhostCost : p.kcost;
    const int Lb_pad = p.nchunk * kColsPerWord;
    const int2 rg = strip_range<kAllCols>(p, strip);  // sub-chunks rg.x .. rg.y-1
    const int n0 = rg.x + half;
    const int q0 = n0 * kSub / S::kBlk;
    br.begin(q0, min((rg.y * kSub + S::kBlk - 1) / S::kBlk, (Lb_pad + S::kBlk - 1) / S::kBlk));
    br.top_up(q0, p.Bhat, Lb_pad, lane);
    int qcur = -1;
    for (int n = n0; n < rg.y; n += Cfg::kNC) {
        const int js = n * kSub;
        const int q = js / S::kBlk;
        if (q != qcur) {
            if (!br.wait(q, p.ctl, p.timeout_ns)) break;
            br.top_up(q, p.Bhat, Lb_pad, lane);
            qcur = q;
        }
        const unsigned t = csub + (unsigned)(n - rg.x);
        const unsigned slot = t % kSlots;
        // the DP warp has read this slot's previous contents
        if (!mbar_wait(bar_at(cempty, slot), use_parity(t, kSlots) ^ 1u, p.ctl, p.timeout_ns, 6))
            break;
        // the 8 frames of the sub-chunk, feature-major (16 floats per feature)
        const unsigned nb = br.chunk_s(js >> 4) + (unsigned)(js & kSub) * 4u;
        float2 c[R][kSub / 2];  // costs of columns 2m, 2m+1 in c[k][m]
#pragma unroll
        for (int k = 0; k < R; ++k)
#pragma unroll
            for (int f = 0; f < kSub / 2; ++f) c[k][f] = make_float2(kc, kc);
        // loads of the next feature group are issued before the FMAs of the
        // current one
        float4 bv[2][2 * kFG];
#pragma unroll
        for (int e = 0; e < kFG; ++e) {
            bv[0][2 * e] = lds128(nb + (unsigned)(e * kColsPerWord) * 4u);
            bv[0][2 * e + 1] = lds128(nb + (unsigned)(e * kColsPerWord + 4) * 4u);
        }
#pragma unroll
        for (int gi = 0; gi < kNG; ++gi) {
            if (gi + 1 < kNG) {
#pragma unroll
                for (int e = 0; e < kFG; ++e) {
                    const int d = (gi + 1) * kFG + e;
                    bv[(gi + 1) & 1][2 * e] = lds128(nb + (unsigned)(d * kColsPerWord) * 4u);
                    bv[(gi + 1) & 1][2 * e + 1] =
                        lds128(nb + (unsigned)(d * kColsPerWord + 4) * 4u);
                }
            }
#pragma unroll
            for (int e = 0; e < kFG; ++e) {
                const int d = gi * kFG + e;
                const float4 b0 = bv[gi & 1][2 * e], b1 = bv[gi & 1][2 * e + 1];
#pragma unroll
                for (int k = 0; k < R; ++k) {
                    const float2 xx = make_float2(na[k][d], na[k][d]);
                    c[k][0] = __ffma2_rn(xx, make_float2(b0.x, b0.y), c[k][0]);
                    c[k][1] = __ffma2_rn(xx, make_float2(b0.z, b0.w), c[k][1]);
                    c[k][2] = __ffma2_rn(xx, make_float2(b1.x, b1.y), c[k][2]);
                    c[k][3] = __ffma2_rn(xx, make_float2(b1.z, b1.w), c[k][3]);
                }
            }
        }
        const unsigned sbase = cring + slot * CR::kSlotBytes;
        const unsigned dst = sbase + (unsigned)lane * 16u;
#pragma unroll
        for (int k = 0; k < R; ++k) {
            sts128(dst + (unsigned)(2 * k) * (kWarp * 16),
                   make_float4(c[k][0].x, c[k][0].y, c[k][1].x, c[k][1].y));
            sts128(dst + (unsigned)(2 * k + 1) * (kWarp * 16),
                   make_float4(c[k][2].x, c[k][2].y, c[k][3].x, c[k][3].y));
        }
        cost_arrive(bar_at(cfull, slot), sbase + CR::kBorder, n, bs, lane);
    }
    br.drain();
}

// Cost warp `half` (of kNC) of `strip` for D > 32, FP32: every kNC-th
// sub-chunk of the strip (those with n - first = half mod kNC), all 8 columns, C' = (1 - mu) - a^_i . b^_j with one FMA per feature in feature
// order (the values of every other decomposition).  A^ of the strip comes
// from the A tile in shared memory (`tile`, 32 R rows of kStride floats),
// which the cost warps of the strip load together at the strip's start
// (named barrier 1 + w), and is reused for 8 columns per load; B^ from the
// warp's own ring of two 16-frame chunks in shared memory, filled by bulk
// copies one chunk ahead (B^ through L1 instead ran at L2 latency, ~1100
// cycles per column; 4 columns per warp and sub-chunk, at 426).  A slot of
// the cost ring is written by one warp, as in the narrow kernel.
template <int DP, int R, int NS, int kSlots>
__device__ __forceinline__ void run_cost_wide(const DpArgs& p, int strip, int w, int half,
                                              int lane, float* tile, unsigned cring,
                                              unsigned cfull, unsigned cempty, unsigned csub,
                                              const BorderSrc& bs,
                                              BRing<DP, CostCfg<DP, NS, false>::kBSlots,
                                                    CostCfg<DP, NS, false>::kBBlk>& br) {
    using W = CostCfg<DP, NS, false>;
    using S = BStage<DP, W::kBSlots, W::kBBlk>;
    using CR = CostRing<R>;
    constexpr int kRows = 31 * R;
    constexpr int kS = W::kStride;
    static_assert(S::kBlk == 2 * kSub, "one chunk of B per sub-chunk pair");
    const bool ghost = lane == kGhostLane;
    // the strip's rows of A^ (ghost rows zero) into the tile, 16 bytes a lane
    {
        constexpr int kT = W::kNC * kWarp;  // the strip's cost warps
        const int tid = half * kWarp + lane;
        for (int e = tid; e < 32 * R * (DP / 4); e += kT) {
            const int r = e / (DP / 4), q = e - r * (DP / 4);
            float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
            if (r < kRows)
                v = reinterpret_cast<const float4*>(p.Ahat + (size_t)(strip * kRows + r) * DP)[q];
            *reinterpret_cast<float4*>(tile + r * kS + 4 * q) = v;
        }
        asm volatile("bar.sync %0, %1;" ::"r"(1 + w), "r"(kT) : "memory");
    }
    const float kc = ghost ? kGhostCost : p.kcost;
    const int Lb_pad = p.nchunk * kColsPerWord;
    const int2 rg = strip_range(p, strip);  // rg.x even: sub-chunk pairs are chunks
    const float* arow = tile + (lane * R) * kS;
    // this warp's sub-chunks n0, n0 + kNC, ...: one in every kNC / 2 chunks of B
    // (kNC is even), which are the blocks 0, 1, ... of its ring
    static_assert(W::kNC % 2 == 0, "a warp keeps to one half of its chunks");
    // groups of 4 features, in whole trips of four: beyond them both frames are
    // zero, and an FMA with a zero product leaves every bit of the sum (24001 x 27011 at
    // D = 100: 3.58 ms, 3.26 so)
    const int ng = min((p.feats + 15) / 16 * 4, DP / 4);
    const int n0 = rg.x + half;
    br.stride = W::kNC / 2;
    br.off = n0 / 2;
    br.begin(0, rg.y > n0 ? (rg.y - n0 + W::kNC - 1) / W::kNC : 0);
    br.top_up(0, p.Bhat, Lb_pad, lane);
    for (int n = n0, q = 0; n < rg.y; n += W::kNC, ++q) {
        if (!br.wait(q, p.ctl, p.timeout_ns)) break;
        br.top_up(q, p.Bhat, Lb_pad, lane);
        // feature d of the sub-chunk's 8 frames: 32 bytes at bsrc + 64 d
        const unsigned bsrc = br.block_s(q) + (unsigned)(n & 1) * 32u;
        const unsigned t = csub + (unsigned)(n - rg.x);
        const unsigned slot = t % kSlots;
        // the DP warp has read this slot's previous contents
        if (!mbar_wait(bar_at(cempty, slot), use_parity(t, kSlots) ^ 1u, p.ctl, p.timeout_ns, 6))
            break;
        // costs of columns 2q, 2q+1 of row k in c[k][q]: each paired FMA is
        // two FP32 FMAs, each rounded once (the values of one FMA per feature
        // in feature order), at half the instructions of scalar FMAs
        float2 c[R][kSub / 2];
#pragma unroll
        for (int k = 0; k < R; ++k)
#pragma unroll
            for (int q = 0; q < kSub / 2; ++q) c[k][q] = make_float2(kc, kc);
        // per group of 4 features: R rows of A^ (one 16-byte load each) and
        // the 8 frames of 4 features of B^ (two 16-byte loads each); two
        // buffers, the next group's loads issued before this group's FMAs
        float4 a0[R], b0[8], a1[R], b1[8];
        auto load = [&](int g, float4* a, float4* b) {
#pragma unroll
            for (int k = 0; k < R; ++k) a[k] = *reinterpret_cast<const float4*>(arow + k * kS + 4 * g);
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                b[2 * e] = lds128(bsrc + (unsigned)(4 * g + e) * 64u);
                b[2 * e + 1] = lds128(bsrc + (unsigned)(4 * g + e) * 64u + 16u);
            }
        };
        auto fmas = [&](const float4* a, const float4* b) {
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const float4 u = b[2 * e], v = b[2 * e + 1];
#pragma unroll
                for (int k = 0; k < R; ++k) {
                    const float x = e == 0 ? a[k].x : (e == 1 ? a[k].y : (e == 2 ? a[k].z : a[k].w));
                    const float2 xx = make_float2(-x, -x);
                    c[k][0] = __ffma2_rn(xx, make_float2(u.x, u.y), c[k][0]);
                    c[k][1] = __ffma2_rn(xx, make_float2(u.z, u.w), c[k][1]);
                    c[k][2] = __ffma2_rn(xx, make_float2(v.x, v.y), c[k][2]);
                    c[k][3] = __ffma2_rn(xx, make_float2(v.z, v.w), c[k][3]);
                }
            }
        };
        // four groups a trip (measured on GB300, one warp alone: 4833 cycles
        // a sub-chunk at D = 128, against 5967 with scalar FMAs and two
        // groups a trip)
        static_assert((DP / 4) % 4 == 0, "whole trips of four feature groups");
        load(0, a0, b0);
#pragma unroll 1
        for (int g = 0; g < ng; g += 4) {
            load(g + 1, a1, b1);
            fmas(a0, b0);
            load(g + 2, a0, b0);
            fmas(a1, b1);
            load(g + 3, a1, b1);
            fmas(a0, b0);
            if (g + 4 < ng) load(g + 4, a0, b0);
            fmas(a1, b1);
        }
        const unsigned sbase = cring + slot * CR::kSlotBytes;
        const unsigned dst = sbase + (unsigned)lane * 16u;
#pragma unroll
        for (int k = 0; k < R; ++k) {
            sts128(dst + (unsigned)(2 * k) * (kWarp * 16),
                   make_float4(c[k][0].x, c[k][0].y, c[k][1].x, c[k][1].y));
            sts128(dst + (unsigned)(2 * k + 1) * (kWarp * 16),
                   make_float4(c[k][2].x, c[k][2].y, c[k][3].x, c[k][3].y));
        }
        cost_arrive(bar_at(cfull, slot), sbase + CR::kBorder, n, bs, lane);
    }
    br.drain();
}

__device__ __forceinline__ void ldsm_x4(unsigned addr, uint32_t& r0, uint32_t& r1, uint32_t& r2,
                                        uint32_t& r3) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];"
                 : "=r"(r0), "=r"(r1), "=r"(r2), "=r"(r3)
                 : "r"(addr)
                 : "memory");
}
// d += a (16x16 bf16, row) * b (16x8 bf16, col), FP32 accumulate.
__device__ __forceinline__ void mma_bf16(float* d, const uint32_t* a, const uint32_t* b) {
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, "
        "{%8, %9}, {%0, %1, %2, %3};"
        : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b[0]), "r"(b[1]));
}
__device__ __forceinline__ uint32_t pack_bf16x2(float lo, float hi) {
    uint32_t r;
    asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(r) : "f"(hi), "f"(lo));
    return r;
}

// BF16 cost warp of `strip` (DP = K = 64 or 128, R = 3 rows per lane): per
// 16 columns one 96 x 16 x DP product on the tensor cores (6 x 2 tiles of
// m16n8k16 per 16 features), costs C' = (1 - mu) - dot written row-major into
// two cost slots; the ghost lane's rows get 1e30.  A's rows are converted to
// bf16 into shared memory once per strip; B's bf16 frames arrive by TMA, one
// chunk per block.
template <int DP, int R, int kNC, int kSlots>
__device__ __forceinline__ void run_cost_bf16(const DpArgs& p, int strip, int w, int half, int lane, unsigned a_s,
                                              unsigned b_s, unsigned bbar_s, unsigned& bbase,
                                              unsigned cring, unsigned cfull, unsigned cempty,
                                              unsigned csub, const BorderSrc& bs) {
    constexpr int kRows = 31 * R;       // real rows of the strip
    constexpr int kM = 32 * R;          // rows of the product (6 tiles of 16)
    constexpr int kMT = kM / 16;
    constexpr int kKS = DP / 16;        // k-steps of 16 features
    constexpr int kRowBytes = kBfStride * 2;
    const int2 rg = strip_range(p, strip);  // sub-chunks rg.x (even) .. rg.y-1
    const int c_lo = rg.x / 2 + half, c_hi = (rg.y + 1) / 2;
    const int nsub = rg.y;
    // A: rows r = 0 .. kM-1 of the strip as bf16 (rows >= kRows are zero)
    for (int r = half * kWarp + lane; r < kM; r += kNC * kWarp) {
        const float* src = p.Ahat + (size_t)(strip * kRows + r) * DP;
#pragma unroll 4
        for (int d = 0; d < DP; d += 8) {
            float4 v0 = make_float4(0.f, 0.f, 0.f, 0.f), v1 = v0;
            if (r < kRows) {
                v0 = *reinterpret_cast<const float4*>(src + d);
                v1 = *reinterpret_cast<const float4*>(src + d + 4);
            }
            const uint32_t w0 = pack_bf16x2(v0.x, v0.y), w1 = pack_bf16x2(v0.z, v0.w);
            const uint32_t w2 = pack_bf16x2(v1.x, v1.y), w3 = pack_bf16x2(v1.z, v1.w);
            asm volatile("st.shared.v4.u32 [%0], {%1, %2, %3, %4};" ::"r"(
                             a_s + (unsigned)(r * kRowBytes + d * 2)),
                         "r"(w0), "r"(w1), "r"(w2), "r"(w3)
                         : "memory");
        }
    }
    if constexpr (kNC > 1)
        asm volatile("bar.sync %0, %1;" ::"r"(1 + w), "r"(kNC * kWarp) : "memory");
    else
        __syncwarp();
    const char* gb = static_cast<const char*>(p.Bbf);
    // this warp's chunks c_lo, c_lo + kNC, ... are the blocks 0 .. nq-1 of its ring
    const int nq = c_hi > c_lo ? (c_hi - c_lo + kNC - 1) / kNC : 0;
    int issued = 0, waited = 0;
    auto issue = [&](int q) {  // lane 0: block q into slot (bbase + q) % kBfSlots
        if (lane == 0) {
            const unsigned t = bbase + (unsigned)q;
            tma_load(b_s + (t % kBfSlots) * kBfBlkBytes,
                     gb + (size_t)(c_lo + q * kNC) * kBfBlkBytes, (unsigned)kBfBlkBytes,
                     bbar_s + 8 * (t % kBfSlots));
        }
    };
    while (issued < nq && issued < kBfSlots - 1) issue(issued++);
    const float kc = p.kcost;
    const int g = lane >> 2, t4 = lane & 3;
    bool ok = true;
    for (int c = c_lo, q = 0; c < c_hi && ok; c += kNC, ++q) {
        // chunk c of B is in its slot
        const unsigned tb = bbase + (unsigned)q;
        if (!mbar_wait(bbar_s + 8 * (tb % kBfSlots), (tb / kBfSlots) & 1u, p.ctl, p.timeout_ns,
                       4)) {
            ok = false;
            break;
        }
        waited = q + 1;
        if (issued < nq) issue(issued++);
        const int nj = (2 * c + 1 < nsub) ? 2 : 1;  // sub-chunks of this chunk
        const unsigned t0 = csub + (unsigned)(2 * c - rg.x);
        for (int j = 0; j < nj; ++j)
            if (!mbar_wait(bar_at(cempty, (t0 + j) % kSlots), use_parity(t0 + j, kSlots) ^ 1u,
                           p.ctl, p.timeout_ns, 6)) {
                ok = false;
                break;
            }
        if (!ok) break;
        // B fragments of the chunk's 16 frames: n-tile j = frames 8j .. 8j+7
        const unsigned bslot = b_s + (tb % kBfSlots) * kBfBlkBytes;
        uint32_t bf[2][kKS][2];
#pragma unroll
        for (int j = 0; j < 2; ++j)
#pragma unroll
            for (int kq = 0; kq < kKS / 2; ++kq)
                ldsm_x4(bslot + (unsigned)((8 * j + (lane & 7)) * kRowBytes +
                                           (32 * kq + 8 * (lane >> 3)) * 2),
                        bf[j][2 * kq][0], bf[j][2 * kq][1], bf[j][2 * kq + 1][0],
                        bf[j][2 * kq + 1][1]);
        float acc[kMT][2][4];
#pragma unroll
        for (int mt = 0; mt < kMT; ++mt)
#pragma unroll
            for (int j = 0; j < 2; ++j)
#pragma unroll
                for (int e = 0; e < 4; ++e) acc[mt][j][e] = 0.f;
#pragma unroll
        for (int mt = 0; mt < kMT; ++mt)
#pragma unroll
            for (int ks = 0; ks < kKS; ++ks) {
                uint32_t a[4];
                ldsm_x4(a_s + (unsigned)((16 * mt + (lane & 7) + 8 * ((lane >> 3) & 1)) *
                                             kRowBytes +
                                         (16 * ks + 8 * (lane >> 4)) * 2),
                        a[0], a[1], a[2], a[3]);
                mma_bf16(acc[mt][0], a, bf[0][ks]);
                mma_bf16(acc[mt][1], a, bf[1][ks]);
            }
        // costs into the two slots: rows 16 mt + g (+8), columns 2 t4, 2 t4 + 1
#pragma unroll
        for (int j = 0; j < 2; ++j) {
            if (j >= nj) break;
            const unsigned slot = cring + ((t0 + j) % kSlots) * CostRingRM<R>::kSlotBytes;
#pragma unroll
            for (int mt = 0; mt < kMT; ++mt) {
                const int r0 = 16 * mt + g, r1 = r0 + 8;
                const float v00 = r0 < kRows ? kc - acc[mt][j][0] : kGhostCost;
                const float v01 = r0 < kRows ? kc - acc[mt][j][1] : kGhostCost;
                const float v10 = r1 < kRows ? kc - acc[mt][j][2] : kGhostCost;
                const float v11 = r1 < kRows ? kc - acc[mt][j][3] : kGhostCost;
                asm volatile("st.shared.v2.f32 [%0], {%1, %2};" ::"r"(
                                 slot + (unsigned)(r0 * kRowFloats * 4 + t4 * 8)),
                             "f"(v00), "f"(v01)
                             : "memory");
                asm volatile("st.shared.v2.f32 [%0], {%1, %2};" ::"r"(
                                 slot + (unsigned)(r1 * kRowFloats * 4 + t4 * 8)),
                             "f"(v10), "f"(v11)
                             : "memory");
            }
            cost_arrive(bar_at(cfull, (t0 + j) % kSlots), slot + CostRingRM<R>::kBorder, 2 * c + j,
                        bs, lane);
        }
    }
    // leave no copy in flight (bounded)
    for (int q = waited; q < issued; ++q) {
        const unsigned tb = bbase + (unsigned)q;
        const long long t0 = __shfl_sync(kFull, global_ns(), 0);
        while (!__all_sync(kFull, mbar_try_wait(bbar_s + 8 * (tb % kBfSlots),
                                                (tb / kBfSlots) & 1u))) {
            if (__shfl_sync(kFull, global_ns(), 0) - t0 > 1000000000LL) break;
        }
    }
    bbase += (unsigned)issued;
}

// Which warps of a CTA a strip group needs: the reader for groups that have
// one above, the writer for groups that have one below.
struct GroupRoles {
    int g, nstrips_here;
    bool reader, writer;
};
template <int NS>
__device__ __forceinline__ GroupRoles group_roles(const DpArgs& p, int g) {
    GroupRoles r;
    r.g = g;
    r.nstrips_here = min(NS, p.nstrips - g * NS);
    r.reader = g > 0;
    r.writer = (g + 1 < p.ngroups) && (g != p.skip_publish);
    return r;
}

// cur[k] for a runtime k < R without indexing the register array.
template <int R>
__device__ __forceinline__ float pick_row(const float* cur, int k) {
    float v = cur[0];
#pragma unroll
    for (int q = 1; q < R; ++q) v = (k == q) ? cur[q] : v;
    return v;
}

// Where a strip's bottom rows go, 8 columns (64 bytes) a block: the border
// part of the next strip's slots, or the writer's ring.  Blocks [first, end)
// are stored, block `first` being lifetime use t0 of the ring.
struct OutRing {
    unsigned base, stride, full, empty, t0;
    int first, end;
};

// A sub-chunk's operands in registers: the lane's costs and the top border's
// (row top-2, row top-1) pairs of two columns per float4.
template <int R>
struct SubIn {
    float4 c[2 * R], g[4];
};
// Load `it` of the 2 R + 4 of a slot.
template <int R, bool kRM>
__device__ __forceinline__ void load_part(SubIn<R>& in, unsigned slot, int lane, int it) {
    if (it < 2 * R) {
        in.c[it] = kRM ? lds128(slot + (unsigned)(lane * R + it / 2) * (kRowFloats * 4) +
                                (unsigned)(it & 1) * 16u)
                       : lds128(slot + (unsigned)lane * 16u + (unsigned)it * (kWarp * 16));
    } else {
        in.g[it - 2 * R] = lds128(slot + SlotOf<R, kRM>::kBorder + (unsigned)(it - 2 * R) * 16u);
    }
}
__device__ __forceinline__ float elem(const float4& v, int k) {
    return k == 0 ? v.x : (k == 1 ? v.y : (k == 2 ? v.z : v.w));
}

// The recurrence state of a strip's lane: columns j-1 and j-2 of its rows and
// row top-1 of column j-2.
template <int R>
struct DpState {
    float cur[R], prv[R], ylp;
};
// Column u of a sub-chunk; behind(): the shared-memory accesses that belong
// behind the column's shuffles (a shuffle waits for the accesses queued before
// it, and the recurrence waits for the shuffles).
template <int R, bool kSubseq, bool kT, class Behind>
__device__ __forceinline__ void sweep_col(const SubIn<R>& in, int u, bool origin, int srcA,
                                          bool ghost, float mu, DpState<R>& s, float* fw,
                                          Behind behind) {
    float cu[R];
#pragma unroll
    for (int k = 0; k < R; ++k) cu[k] = elem(in.c[2 * k + u / 4], u & 3);
    const float y1 = __shfl_sync(kFull, s.cur[R - 1], srcA);  // E[i0-1][j-1]
    const float y2 = __shfl_sync(kFull, s.cur[R - 2], srcA);  // E[i0-2][j-1]
    behind();
    dp_cells<R, kSubseq, kT>(cu, u, y1, y2, ghost, elem(in.g[u / 2], 2 * (u & 1)),
                             elem(in.g[u / 2], 2 * (u & 1) + 1), origin, mu, s.cur, s.prv, s.ylp,
                             fw);
}

// DP warp of `strip`: sub-chunks rg of its slots (cring, cfull, cempty, the
// first being lifetime use csub), the bottom rows into `out`.
//
// What bounds it: one warp's chain of columns (a column's two shuffles, FMAs
// and minima feed the next column's shuffles, two columns apart at R = 3), and
// with it the chain of strips.  Alone on an SM sub-partition 16 columns of
// straight-line code take ~43 cycles a column; every branch between columns
// costs ~50 cycles (the fields of the last columns no longer overlap the next
// ones), and waits, loads and stores that stand between sub-chunks cost more.
// So a trip of the loop is a backpointer word (sub-chunks n and n + 1) with one
// branch: it starts with the operands of n in registers, loads those of n + 1
// and n + 2 behind the shuffles after testing their barriers, sweeps n + 1
// before knowing that its operands were there, and looks at all tests at its
// end.  Where they were not, the state before n + 1 is put back, the barrier is
// waited for and n + 1 is swept again: in a chain that is on time this is
// rare, and a strip that is early has time to lose.
template <int R, int NS, int kSlots, bool kRM, bool kSubseq, bool kT>
__device__ __forceinline__ void run_dp(const DpArgs& p, int strip, int lane, const int2 rg,
                                       const OutRing& out, unsigned cring, unsigned cfull,
                                       unsigned cempty, unsigned csub) {
    using Slot = SlotOf<R, kRM>;
    constexpr int kRows = 31 * R;
    constexpr int kLoads = 2 * R + 4;  // 16-byte loads of a slot
    // the next slot's barrier is tested behind the shuffles of column kTest and the slot
    // loaded behind those of columns kFirst, kFirst + 1, .., kPer loads each: as late
    // as the latencies allow, since a strip can follow the one above no closer than
    // its tests look ahead (20000 x 25000, D = 12: DP 0.907 ms, 0.947 a column
    // earlier; 40000 x 48000 with the BF16 cost 2.445, 2.437)
    constexpr int kTest = 4, kFirst = 5, kPer = 4;
    const bool ghost = lane == kGhostLane;
    const int i0 = strip * kRows + lane * R;
    const float mu = p.mu;
    const int srcA = (lane + 31) & 31;
    const bool is_origin = (i0 == 0) && !ghost;
    // subsequence DP: the lane and row slot of row La-1, if this strip holds it
    const int rl = p.La - 1 - strip * kRows;
    const bool has_last = kSubseq && rl >= 0 && rl < kRows && lane == rl / R;
    const int kl = kSubseq ? rl - (rl / R) * R : 0;
    const int nfull = min(rg.y, p.Lb / kSub);  // sub-chunks before it have all 8 columns

    DpState<R> s;
#pragma unroll
    for (int k = 0; k < R; ++k) s.cur[k] = s.prv[k] = INFINITY;
    s.ylp = INFINITY;

    auto wait_load = [&](unsigned t, SubIn<R>& in) -> bool {
        if (!mbar_wait(bar_at(cfull, t % kSlots), use_parity(t, kSlots), p.ctl, p.timeout_ns, 7))
            return false;
#pragma unroll
        for (int it = 0; it < kLoads; ++it)
            load_part<R, kRM>(in, cring + (t % kSlots) * Slot::kBytes, lane, it);
        return true;
    };
    auto release = [&](unsigned t) {
        __syncwarp();
        mbar_arrive_if(bar_at(cempty, t % kSlots), lane == 0);
    };
    // The 8 columns of a full sub-chunk: fields into word's half h, the bottom
    // rows to dst where st holds; behind(u): see sweep_col.  (No poll of the
    // failure flag in the sweep: every wait checks it on its slow path, and a
    // warp that never waits ends with its strip.)
    auto full_sub = [&](int n, const SubIn<R>& in, int h, unsigned dst, bool st, uint32_t* word,
                        auto behind) {
        float fw[R];  // backpointer fields of the sub-chunk, bits 2u, 2u+1
#pragma unroll
        for (int k = 0; k < R; ++k) fw[k] = 0.0f;
        float ol[kSub];  // subsequence DP: row La-1 (lane of has_last)
        (void)ol;
#pragma unroll
        for (int u = 0; u < kSub; ++u) {
            sweep_col<R, kSubseq, kT>(
                in, u, (kSubseq || (h == 0 && u == 0 && n == 0)) && is_origin, srcA, ghost, mu, s,
                fw, [&] {
                    if (u > 0)
                        sts64_if(dst + (unsigned)(u - 1) * 8u, s.cur[R - 2], s.cur[R - 1], st);
                    behind(u);
                });
            if constexpr (kSubseq) ol[u] = pick_row<R>(s.cur, kl);
        }
        sts64_if(dst + (unsigned)(kSub - 1) * 8u, s.cur[R - 2], s.cur[R - 1], st);
        if constexpr (kSubseq) {  // row La-1 of these columns
            float* d = p.lastrow + n * kSub;
            stg128_if(d, ol[0], ol[1], ol[2], ol[3], has_last);
            stg128_if(d + 4, ol[4], ol[5], ol[6], ol[7], has_last);
        }
#pragma unroll
        for (int k = 0; k < R; ++k) word[k] |= field_bits(fw[k], h);
    };
    // the loads of a slot behind the shuffles of columns kFirst, kFirst + 1, ...
    auto part = [&](SubIn<R>& in, unsigned slot, int u) {
        if (u >= kFirst) {
#pragma unroll
            for (int z = 0; z < kPer; ++z)
                if (kPer * (u - kFirst) + z < kLoads)
                    load_part<R, kRM>(in, slot, lane, kPer * (u - kFirst) + z);
        }
    };
    // Whether use t is there, and the slot to load next: its own, or where it is not yet
    // there that of use t - 1, whose values are then dropped.  The address comes
    // from the test's result, so that no load can be performed before the test.  (Loads of
    // use t's slot in any case, dropped like these where the test failed, came too early
    // now and then: with six cost warps a strip at D = 100 one call in 70 of 12007 x 9001
    // frames had a wrong total; since then none in 23000.)
    auto slot_of = [&](unsigned t) { return cring + (t % kSlots) * Slot::kBytes; };
    auto test = [&](unsigned t, int& there) -> unsigned {
        there = mbar_test_wait(bar_at(cfull, t % kSlots), use_parity(t, kSlots));
        return slot_of(there ? t : t - 1u);
    };
    // The trip's end takes the outcomes from the tests in the FP32 cluster kernels and with
    // four strips a CTA, and elsewhere from the slots that were loaded, which keeps two
    // registers less (DP of 20000 x 25000 at D = 12, in clusters: 0.907 ms, 0.950 from the
    // slots; of 256 pairs, four strips a CTA, 3.225 and 3.254; the whole call of 40000 x 48000
    // with the BF16 cost 2.80 and 2.72, of 256 planned pairs 3.53 and 3.51, of 32 fragments of
    // 40003 x 50021 frames 4.27 and 4.11).
    constexpr bool kKeepTests = (kSlots > 8 && !kRM) || NS == 4;
    auto store = [&](int n, uint32_t* word) {
        if constexpr (kT) {
#pragma unroll
            for (int k = 0; k < R; ++k) word[k] = transpose_fields(word[k]);
        }
        store_words<R>(p.bp + ((size_t)strip * p.nchunk + (size_t)(n >> 1)) * (32 * R) +
                           (size_t)lane * R,
                       word);
    };

    int n = rg.x;  // even: ranges start on whole words
    unsigned t = csub;
    SubIn<R> ia, ib;
    if (!wait_load(t, ia)) return;
    release(t);
#pragma unroll 1
    for (; n + 1 < nfull; n += 2, t += 2) {
        uint32_t word[R], wordb[R];
#pragma unroll
        for (int k = 0; k < R; ++k) word[k] = wordb[k] = 0u;
        // out.first is even too; blocks n and n + 1 of the output ring are free
        // (those of a group's first trips, later ones by the test below)
        const bool on = n >= out.first && n < out.end;
        const bool st = on && lane == kOutLane;
        const bool more = n + 2 < rg.y;
        const bool next_on = n + 2 >= out.first && n + 2 < out.end;
        const unsigned to = out.t0 + (unsigned)(n - out.first);
        const unsigned dst0 = out.base + (to % kSlots) * out.stride;
        const unsigned dst1 = out.base + ((to + 1u) % kSlots) * out.stride;
        int rb = 1, ra = 1, ro = 1;
        unsigned sb = 0, sa = 0;  // the slots loaded
        full_sub(n, ia, 0, dst0, st, word, [&](int u) {
            if (u == kTest) sb = test(t + 1u, rb);
            part(ib, sb, u);
        });
        mbar_arrive_if(bar_at(out.full, to % kSlots), st);
        const DpState<R> before = s;
        full_sub(n + 1, ib, 1, dst1, st, wordb, [&](int u) {
            if (u == 0)  // its consumer empties the output ring in order
                ro = mbar_test_wait(bar_at(out.empty, (to + 3u) % kSlots),
                                    use_parity(to + 3u, kSlots) ^ 1u);
            if (u == kTest) sa = test(t + 2u, ra);
            part(ia, sa, u);
        });
        int go;  // (a vote on whole numbers, or on predicates: 0.907 and 1.009 ms in clusters)
        if constexpr (kKeepTests)
            go = __all_sync(kFull, rb & (ra | (int)!more) & (ro | (int)!next_on));
        else
            go = __all_sync(kFull, (sb == slot_of(t + 1u)) & ((sa == slot_of(t + 2u)) | !more) &
                                       ((bool)ro | !next_on));
        if (!go) {
            if (!__all_sync(kFull, kKeepTests ? rb : (int)(sb == slot_of(t + 1u)))) {
                if (!wait_load(t + 1u, ib)) return;
                s = before;
#pragma unroll
                for (int k = 0; k < R; ++k) wordb[k] = 0u;
                full_sub(n + 1, ib, 1, dst1, st, wordb, [](int) {});
            }
            // nothing is held back while this warp waits: what feeds the next
            // slot may itself wait for this one's release
            mbar_arrive_if(bar_at(out.full, (to + 1u) % kSlots), st);
            release(t + 1u);
            if (more && !wait_load(t + 2u, ia)) return;
            if (next_on && !mbar_wait(bar_at(out.empty, (to + 3u) % kSlots),
                                      use_parity(to + 3u, kSlots) ^ 1u, p.ctl, p.timeout_ns, 2))
                return;
            __syncwarp();
        } else {
            mbar_arrive_if(bar_at(out.full, (to + 1u) % kSlots), st);
            release(t + 1u);
        }
        mbar_arrive_if(bar_at(cempty, (t + 2u) % kSlots), lane == 0 && more);
#pragma unroll
        for (int k = 0; k < R; ++k) word[k] |= wordb[k];
        store(n, word);
    }
    // up to two sub-chunks are left: a full one without a partner, and the
    // ragged one at the end of B; one at a time
    if (n < rg.y) {
        uint32_t word[R];
#pragma unroll
        for (int k = 0; k < R; ++k) word[k] = 0u;
        const int n0 = n;
#pragma unroll 1
        for (; n < rg.y; ++n, ++t) {
            const int nsteps = min(kSub, p.Lb - n * kSub);
            const bool on = n >= out.first && n < out.end;
            const unsigned to = out.t0 + (unsigned)(n - out.first);
            if (on && !mbar_wait(bar_at(out.empty, to % kSlots), use_parity(to, kSlots) ^ 1u, p.ctl,
                                 p.timeout_ns, 2))
                return;
            const bool st = on && lane == kOutLane;
            const unsigned dst = out.base + (to % kSlots) * out.stride;
            float fw[R];
#pragma unroll
            for (int k = 0; k < R; ++k) fw[k] = 0.0f;
#pragma unroll
            for (int u = 0; u < kSub; ++u) {
                if (u >= nsteps) break;
                sweep_col<R, kSubseq, kT>(ia, u, (kSubseq || (n == 0 && u == 0)) && is_origin, srcA,
                                          ghost, mu, s, fw, [] {});
                sts64_if(dst + (unsigned)u * 8u, s.cur[R - 2], s.cur[R - 1], st);
                if constexpr (kSubseq)
                    if (has_last) p.lastrow[n * kSub + u] = pick_row<R>(s.cur, kl);
            }
            mbar_arrive_if(bar_at(out.full, to % kSlots), st);
#pragma unroll
            for (int k = 0; k < R; ++k) word[k] |= field_bits(fw[k], 0) << (16 * (n - n0));
            if (n + 1 < rg.y) {
                if (!wait_load(t + 1u, ia)) return;
                release(t + 1u);
            }
        }
        store(n0, word);
    }
#pragma unroll
    for (int k = 0; k < R; ++k)
        if (!ghost && i0 + k == p.La - 1) *p.e_final = s.cur[k];
}

// Reader warp (groups g > 0): the bottom rows of group g-1 from the global
// border into the border part of the first strip's slots.  Lane v < 16 carries
// value v of every sub-chunk (column v / 2, row top-2 + v % 2); loads run
// kAheadSub sub-chunks ahead, and a value whose tag is not yet this call's is
// re-polled (bounded).  grow: the row of the global border (one per group, in a
// cluster one per ticket: only its last CTA publishes there).
constexpr int kAheadSub = 4;
template <int kSlots>
__device__ __forceinline__ void run_reader(const DpArgs& p, int grow, int lane, unsigned border,
                                           unsigned stride, unsigned full, unsigned empty,
                                           unsigned csub, int nfirst, int nsub, int clo, int chi) {
    // blocks nfirst .. nsub-1 (this group's first strip's range); only columns
    // clo .. chi-1 were published above (the others read as +inf)
    const int Lb = p.Lb;
    clo = max(clo, 0);
    chi = min(chi, Lb);
    const unsigned long long* gin = p.gborder + (size_t)grow * Lb * 2;
    const unsigned epoch = p.epoch;
    const bool act_lane = lane < 2 * kSub;
    const int cofs = (lane >> 1) & (kSub - 1), row = lane & 1;
    unsigned long long pend[kAheadSub];
#pragma unroll
    for (int q = 0; q < kAheadSub; ++q) {
        const int col = (nfirst + q) * kSub + cofs;
        pend[q] = (act_lane && col >= clo && col < chi) ? ldg1(gin + (size_t)col * 2 + row) : 0ull;
    }
    for (int n0 = nfirst; n0 < nsub; n0 += kAheadSub) {
#pragma unroll
        for (int q = 0; q < kAheadSub; ++q) {
            const int n = n0 + q;
            if (n >= nsub) break;
            const int col = n * kSub + cofs;
            const bool act = act_lane && col >= clo && col < chi;
            int ok = !act || tag_of(pend[q]) == epoch;
            if (!__all_sync(kFull, ok)) {
                // each poll is a round trip to L2; status and deadline every 16 polls
                const long long t0 = __shfl_sync(kFull, global_ns(), 0);
                for (int poll = 1;; ++poll) {
                    if (!ok) {
                        pend[q] = ldg1(gin + (size_t)col * 2 + row);
                        ok = tag_of(pend[q]) == epoch;
                    }
                    if (__all_sync(kFull, ok)) break;
                    if ((poll & 15) == 0) {
                        if (__shfl_sync(kFull, read_status(p.ctl), 0) != 0) return;
                        const long long now = __shfl_sync(kFull, global_ns(), 0);
                        if (now - t0 > p.timeout_ns) {
                            if (lane == 0) raise_status(p.ctl, DTW_ERR_TIMEOUT, 3);
                            return;
                        }
                    }
                }
            }
            const unsigned t = csub + (unsigned)(n - nfirst);
            if (!mbar_wait(bar_at(empty, t % kSlots), use_parity(t, kSlots) ^ 1u, p.ctl,
                           p.timeout_ns, 8))
                return;
            if (act_lane)
                sts32(border + (t % kSlots) * stride + (unsigned)lane * 4u,
                      act ? val_of(pend[q]) : INFINITY);
            __syncwarp();
            mbar_arrive_if(bar_at(full, t % kSlots), lane == 0);
            const int ncol = col + kAheadSub * kSub;
            if (act_lane && ncol >= clo && ncol < chi) pend[q] = ldg1(gin + (size_t)ncol * 2 + row);
        }
    }
}

// Writer warp: the last strip's bottom rows from the writer's ring to the
// global border of group g, as (value, epoch) words; lanes 0..15 store one
// coalesced 128-byte line per sub-chunk.
template <int kSlots>
__device__ __forceinline__ void run_writer(const DpArgs& p, int grow, int lane,
                                           const float (*ringo)[2 * kSub], unsigned bfullo,
                                           unsigned bemptyo, unsigned rbase, int nfirst,
                                           int nsub) {
    const int Lb = p.Lb;
    unsigned long long* gout = p.gborder + (size_t)grow * Lb * 2;
    const unsigned epoch = p.epoch;
    for (int n = nfirst; n < nsub; ++n) {
        const unsigned t = rbase + (unsigned)(n - nfirst);
        if (!mbar_wait(bar_at(bfullo, t % kSlots), use_parity(t, kSlots), p.ctl, p.timeout_ns, 9))
            return;
        const float v = ringo[t % kSlots][lane & (2 * kSub - 1)];
        const int col = n * kSub + ((lane >> 1) & (kSub - 1));
        if (lane < 2 * kSub && col < Lb) stg1(gout + (size_t)col * 2 + (lane & 1), pack(v, epoch));
        __syncwarp();
        mbar_arrive_if(bar_at(bemptyo, t % kSlots), lane == 0);
    }
}

// Writer warp of a CTA with another CTA of its cluster below: the blocks of
// the last strip's range [nfirst, nsub) from the writer's ring into the slots
// of the first strip of CTA crank + 1, whose range starts at block bfirst with
// lifetime use bsub of its slots; each of the 16 values an asynchronous store
// completing 4 of the 64 bytes the slot's full barrier expects.  (Blocks before
// bfirst are not needed below.)  The reader warp below hands the slots back in pages
// of kLinkPage uses on `lempty`: page q of the ticket is page lsub + q of the link, and
// its first store waits until page lsub + q - kSlots / kLinkPage is back, which holds
// its slots' previous uses where they lie in this ticket (those of earlier
// tickets are all released).
template <int kSlots>
__device__ __forceinline__ void run_link_writer(const DpArgs& p, int lane,
                                                const float (*ringo)[2 * kSub], unsigned bfullo,
                                                unsigned bemptyo, unsigned rbase, int nfirst,
                                                int nsub, unsigned border, unsigned stride,
                                                unsigned full, unsigned lempty, unsigned lsub,
                                                unsigned bsub, int bfirst, unsigned crank) {
    // peer addresses (a CTA's window of the cluster's shared memory is linear)
    const unsigned rborder = map_rank(border, crank + 1) + (unsigned)lane * 4u;
    const unsigned rfull = map_rank(full, crank + 1);
    for (int n = nfirst; n < nsub; ++n) {
        const unsigned t = rbase + (unsigned)(n - nfirst);  // use of the writer's ring
        const unsigned u = bsub + (unsigned)(n - bfirst);   // use of the slots below
        const bool send = n >= bfirst;
        if (send && (n - bfirst) % kLinkPage == 0) {
            constexpr unsigned kPages = kSlots / kLinkPage;
            const unsigned pg = lsub + (unsigned)(n - bfirst) / kLinkPage;
            // the slots below are normally free long before the block is there
            if (!mbar_wait(bar_at(lempty, pg % kPages), use_parity(pg, kPages) ^ 1u, p.ctl,
                           p.timeout_ns, 10))
                return;
        }
        if (!mbar_wait(bar_at(bfullo, t % kSlots), use_parity(t, kSlots), p.ctl, p.timeout_ns, 9))
            return;
        const float v = ringo[t % kSlots][lane & (2 * kSub - 1)];
        if (send && lane < 2 * kSub)
            st_async_f32(rborder + (u % kSlots) * stride, v, bar_at(rfull, u % kSlots));
        __syncwarp();
        mbar_arrive_if(bar_at(bemptyo, t % kSlots), lane == 0);
    }
}

// Reader warp of a CTA with another CTA of its cluster above: the first
// strip's blocks [nfirst, nsub), uses csub .. of its slots.  Those the CTA above
// sends (before nsent; pages lsub .. of the link) it hands back, kLinkPage at a time,
// once the DP warp has released their slots; the later ones read +inf.  (It also stores those,
// rather than the cost warp, so that no slot can be released twice before
// this warp has seen the first release.)
template <int kSlots>
__device__ __forceinline__ void run_link_reader(const DpArgs& p, int lane, unsigned border,
                                                unsigned stride, unsigned full, unsigned empty,
                                                unsigned csub, int nfirst, int nsent, int nsub,
                                                unsigned lempty, unsigned lsub, unsigned crank) {
    for (int n = nfirst; n < nsub; ++n) {
        const unsigned t = csub + (unsigned)(n - nfirst), slot = t % kSlots;
        if (n < nsent) {
            if (!mbar_wait(bar_at(empty, slot), use_parity(t, kSlots), p.ctl, p.timeout_ns, 11))
                return;
            if ((n - nfirst) % kLinkPage == kLinkPage - 1 || n + 1 == nsent) {
                const unsigned pg = lsub + (unsigned)(n - nfirst) / kLinkPage;
                if (lane == 0)
                    mbar_arrive_remote(map_rank(bar_at(lempty, pg % (kSlots / kLinkPage)), crank - 1));
                __syncwarp();
            }
        } else {
            if (!mbar_wait(bar_at(empty, slot), use_parity(t, kSlots) ^ 1u, p.ctl, p.timeout_ns, 8))
                return;
            if (lane < 2 * kSub) sts32(border + slot * stride + (unsigned)lane * 4u, INFINITY);
            __syncwarp();
            mbar_arrive_if(bar_at(full, slot), lane == 0);
        }
    }
}

// NS strips per CTA: per strip its DP warp and kNC cost warps, and a reader and
// a writer warp (their places: see `role`).  Persistent: a CTA takes strip
// groups from the ticket counter until none are left, so a group only ever
// waits on groups that started earlier.
// kMany: the groups come from a work queue over many pairs (`many`, `items`,
// `ticket`; see launch_dp_split_many) instead of the pair `one`.
// kCl (one pair): the kernel runs in clusters of cn CTAs that
// take tickets together: ticket T gives CTA rank r the strip group
// T cn + r, so the border between two of a ticket's groups goes through
// distributed shared memory (run_link_writer, run_link_reader); only rank 0
// reads a global border and only rank cn - 1 writes one.  A CTA leaves only
// when its whole cluster does (no CTA's shared memory may disappear while a
// peer can still reach it).
template <int DP, int R, int NS, bool kMany, bool kBF, bool kSubseq = false, bool kT = false,
          bool kCl = false>
__global__ void __launch_bounds__(split_threads<DP, NS, kBF>(),
                                  (kCl ? 1 : split_ctas_per_sm(R, NS, DP, kBF)))
    k_dp_split(const DpArgs one, const DpArgs* __restrict__ many, const int2* __restrict__ items,
               int nitems, int* ticket) {
    static_assert(!kCl || (!kMany && !kSubseq), "clusters sweep one plain pair");
    constexpr int kThreads = split_threads<DP, NS, kBF>();
    using Cfg = CostCfg<DP, NS, kBF>;
    constexpr int kSlots = slots_of<kCl>();
    using M = SplitSmem<DP, R, NS, kBF, kCl>;
    using Slot = SlotOf<R, kBF>;
    constexpr int kNC = Cfg::kNC;  // cost warps per strip
    constexpr int kBars = kBF ? kBfSlots : Cfg::kBSlots;
    __shared__ __align__(16) float ringo[kSlots][2 * kSub];  // the writer's ring
    __shared__ __align__(8) unsigned long long bbar[NS * kNC][kBars];
    __shared__ __align__(8) unsigned long long cfull[NS][kSlots];
    __shared__ __align__(8) unsigned long long cempty[NS][kSlots];
    __shared__ __align__(8) unsigned long long ofull[kSlots];
    __shared__ __align__(8) unsigned long long oempty[kSlots];
    // releases of the slots of the CTA below, in a cluster
    __shared__ __align__(8) unsigned long long lempty[kSlots / kLinkPage];
    __shared__ int s_group, s_pair;
    extern __shared__ __align__(128) unsigned char dyn[];  // NS * M::kStripBytes
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const unsigned crank = kCl ? cluster_rank() : 0u;
    const unsigned cn = kCl ? cluster_size() : 1u;
    // Warp roles by SM sub-partition (warp w runs on sub-partition w % 4).  Two
    // cost warps a strip: the DP warps (0, 1) share theirs with the reader and
    // the writer (4, 5) only, the cost warps (2, 3 and 6, 7) have the other two
    // (a DP warp beside a cost warp: 136 against 111 cycles a column on the
    // 20000 x 25000 pair).  One cost warp a strip: the cost warps, the DP warps,
    // then the reader and the writer.
    int role, w = 0, half = 0;
    if (NS == 1) {
        role = wid == 0 ? 1 : (wid == 4 ? 2 : (wid == 5 ? 3 : 0));
        half = wid < 4 ? wid - 1 : wid - 3;
    } else if (NS == 2 && kNC >= 2) {
        role = wid < 2 ? 1 : (wid == 4 ? 2 : (wid == 5 ? 3 : 0));
        if (role < 2) w = wid & 1;
        half = wid < 4 ? 0 : wid / 2 - 2;
    } else {
        role = wid < kNC * NS ? 0 : (wid < (kNC + 1) * NS ? 1 : (wid == (kNC + 1) * NS ? 2 : 3));
        if (role < 2) w = role == 0 ? wid % NS : wid - kNC * NS;
        half = role == 0 ? wid / NS : 0;
    }
    unsigned char* mine = dyn + (size_t)w * M::kStripBytes;
    const unsigned cring_s = smem_u32(mine + M::kOperandBytes);
    const unsigned a_s = smem_u32(mine);                                  // kBF: A tile
    const unsigned b_s = smem_u32(mine + 32 * R * kBfStride * 2 + half * kBfSlots * kBfBlkBytes);  // kBF: B ring
    unsigned bbase = 0;  // kBF: lifetime count of this cost warp's B blocks
    const unsigned cfull_s = smem_u32(&cfull[w][0]);
    const unsigned cempty_s = smem_u32(&cempty[w][0]);

    // the FP32 cost warps' rings of B: behind the A tile where there is one
    BRing<DP, Cfg::kBSlots, Cfg::kBBlk> br;
    br.stage_s = smem_u32(mine + (Cfg::kWide ? 32 * R * Cfg::kStride * 4 : 0) +
                          half * BStage<DP, Cfg::kBSlots, Cfg::kBBlk>::kWarpBytes);
    br.stage = reinterpret_cast<const float*>(mine);  // (not read through this pointer)
    br.bar_s = smem_u32(&bbar[half * NS + w][0]);
    br.base = 0;
    br.first = 0;
    br.nblk = 0;
    br.issued = br.waited = 0;
    if (threadIdx.x == 0) {
        for (int s = 0; s < NS * kNC; ++s)
            for (int k = 0; k < kBars; ++k) mbar_init(smem_u32(&bbar[s][k]), 1);
        for (int k = 0; k < kSlots; ++k) {
            for (int s = 0; s < NS; ++s) {
                mbar_init(smem_u32(&cfull[s][k]), 2);   // the slot's costs, its border
                mbar_init(smem_u32(&cempty[s][k]), 1);  // the DP warp
            }
            mbar_init(smem_u32(&ofull[k]), 1);   // lane 30 of the last strip's DP warp
            mbar_init(smem_u32(&oempty[k]), 1);  // the writer
            if (kCl && k < kSlots / kLinkPage)
                mbar_init(smem_u32(&lempty[k]), 1);  // the reader of the CTA below
        }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if constexpr (kCl) {
        chain_wait();  // for the normalised sequences and ctl
        asm volatile("fence.proxy.async;" ::: "memory");  // the bulk copies read them, too
        chain_next();
        cluster_sync_all();  // every CTA's barriers before any remote access
    }
    // Lifetime sub-chunk counts of the slots and of the writer's ring, and (in
    // a cluster) of the slots of the first strip of the CTA below; page counts of the
    // links into and out of this CTA.
    unsigned csub[NS], osub = 0, lsub = 0, lin = 0, lout = 0;
#pragma unroll
    for (int s = 0; s < NS; ++s) csub[s] = 0;

    for (;;) {
        if constexpr (kCl) {
            // every warp of the cluster finished the previous ticket; rank 0
            // takes the next one and hands it to every CTA of the cluster
            cluster_sync_all();
            if (crank == 0 && threadIdx.x == 0) {
                const int T = read_status(one.ctl) != 0 ? one.ngroups
                                                        : atomicAdd(&one.ctl->ticket, 1);
                for (unsigned r = 0; r < cn; ++r)
                    st_cluster_u32(map_rank(smem_u32(&s_pair), r), (unsigned)T);
            }
            cluster_sync_all();
            const int T = s_pair;
            if ((long long)T * cn >= one.ngroups) break;  // the whole cluster leaves
            if (threadIdx.x == 0) s_group = T * (int)cn + (int)crank;
        } else {
            __syncthreads();  // every warp finished the previous group
        }
        if (!kCl && threadIdx.x == 0) {
            if (kMany) {
                const int t = atomicAdd(ticket, 1);
                int pi = -1, gi = 0;
                if (t < nitems) {
                    pi = items[t].x;
                    // nothing of a failed pair runs
                    gi = read_status(many[pi].ctl) != 0 ? -1 : items[t].y;
                }
                s_pair = pi;
                s_group = gi;
            } else {
                s_pair = 0;
                s_group = read_status(one.ctl) != 0 ? one.ngroups
                                                    : atomicAdd(&one.ctl->ticket, 1);
            }
        }
        __syncthreads();
        if (kMany && s_pair < 0) return;
        if (kMany && s_group < 0) continue;
        const DpArgs p = kMany ? many[s_pair] : one;
        const int g = s_group;
        if (kCl && g >= p.ngroups) continue;  // this CTA's group of the ticket does not exist
        if (g >= p.ngroups) return;
        const GroupRoles gr = group_roles<NS>(p, g);
        const int strip = g * NS + w;
        // the sub-chunk ranges of the group's strips, and of the strips above
        // and below the group
        int2 rgs[NS];
#pragma unroll
        for (int q = 0; q < NS; ++q)
            rgs[q] = q < gr.nstrips_here ? strip_range<kSubseq>(p, g * NS + q) : make_int2(0, 0);
        const int2 above = g > 0 ? strip_range<kSubseq>(p, g * NS - 1) : make_int2(0, 0);
        const int2 below = g + 1 < p.ngroups ? strip_range<kSubseq>(p, (g + 1) * NS) : make_int2(0, 0);
        const bool link_in = kCl && crank > 0, link_out = kCl && crank + 1 < cn;
        int2 rg = rgs[0], rup = above, rdown = below;  // of strip slot w and its neighbours
        unsigned cs = csub[0], cs_down = 0;
#pragma unroll
        for (int q = 0; q < NS; ++q)
            if (q == w) {
                rg = rgs[q];
                cs = csub[q];
                if (q > 0) rup = rgs[q - 1];
                if (q + 1 < NS) {
                    rdown = rgs[q + 1 < NS ? q + 1 : q];
                    cs_down = csub[q + 1 < NS ? q + 1 : q];
                }
            }
        if (role == 0) {
            if (w < gr.nstrips_here) {
                // the border: from the strip above; none above strip 0; for the
                // first strip the reader warp fills in what the group above lacks
                BorderSrc bs;
                bs.inf_from = strip == 0 ? 0 : (w > 0 ? rup.y : 0x7fffffff);
                bs.link_end = w == 0 && g > 0 && link_in ? rup.y : 0;
                if constexpr (kBF)
                    run_cost_bf16<DP, R, kNC, kSlots>(p, strip, w, half, lane, a_s, b_s,
                                                      smem_u32(&bbar[half * NS + w][0]), bbase,
                                         cring_s, cfull_s, cempty_s, cs, bs);
                else if constexpr (Cfg::kWide)
                    run_cost_wide<DP, R, NS, kSlots>(p, strip, w, half, lane, reinterpret_cast<float*>(mine),
                                         cring_s, cfull_s, cempty_s, cs, bs, br);
                else if constexpr (DP > 16 && NS > 1) {
                    // groups of four features that are padding in both frames are left out:
                    // an FMA with a zero product leaves every bit of the sum.  A loop for each
                    // number of groups, as a test in one loop costs D = 32 3%: DP of 48 pairs of up
                    // to 2500 frames, 5 to 8 groups: 177, 185, 192, 205 us, all as 8 before.
                    // With one strip a CTA the cost warps don't set the pace.
                    if (p.feats > 28)
                        run_cost<DP, R, NS, kSlots, kSubseq, 8>(p, strip, half, lane, cring_s, cfull_s,
                                                                cempty_s, cs, bs, br);
                    else if (p.feats > 24)
                        run_cost<DP, R, NS, kSlots, kSubseq, 7>(p, strip, half, lane, cring_s, cfull_s,
                                                                cempty_s, cs, bs, br);
                    else if (p.feats > 20)
                        run_cost<DP, R, NS, kSlots, kSubseq, 6>(p, strip, half, lane, cring_s, cfull_s,
                                                                cempty_s, cs, bs, br);
                    else
                        run_cost<DP, R, NS, kSlots, kSubseq, 5>(p, strip, half, lane, cring_s, cfull_s,
                                                                cempty_s, cs, bs, br);
                } else
                    run_cost<DP, R, NS, kSlots, kSubseq>(p, strip, half, lane, cring_s,
                                                                cfull_s, cempty_s, cs, bs, br);
            }
        } else if (role == 1) {
            if (w < gr.nstrips_here) {
                OutRing out;
                if (w + 1 < NS && w + 1 < gr.nstrips_here) {
                    // the next strip's slots: its blocks, as far as this strip has them
                    out.base = cring_s + (unsigned)M::kStripBytes + Slot::kBorder;
                    out.stride = Slot::kBytes;
                    out.full = cfull_s + 8u * kSlots;
                    out.empty = cempty_s + 8u * kSlots;
                    out.t0 = cs_down;
                    out.first = rdown.x;
                    out.end = rg.y;
                } else {
                    out.base = smem_u32(&ringo[0][0]);
                    out.stride = kBorderBytes;
                    out.full = smem_u32(&ofull[0]);
                    out.empty = smem_u32(&oempty[0]);
                    out.t0 = osub;
                    out.first = rg.x;
                    out.end = w == NS - 1 && gr.writer ? rg.y : rg.x;
                }
                run_dp<R, NS, kSlots, kBF, kSubseq, kT>(p, strip, lane, rg, out, cring_s, cfull_s,
                                                    cempty_s, cs);
            }
        } else if (role == 2) {
            if (gr.reader) {
                if (link_in)
                    run_link_reader<kSlots>(p, lane, cring_s + Slot::kBorder, Slot::kBytes, cfull_s,
                                    cempty_s, csub[0], rgs[0].x, above.y, rgs[0].y,
                                    smem_u32(&lempty[0]), lin, crank);
                else
                    run_reader<kSlots>(p, kCl ? (g - 1) / (int)cn : g - 1, lane, cring_s + Slot::kBorder, Slot::kBytes, cfull_s, cempty_s,
                               csub[0], rgs[0].x, rgs[0].y, above.x * kSub, above.y * kSub);
            }
        } else {
            if (gr.writer) {
                if (link_out)
                    run_link_writer<kSlots>(p, lane, ringo, smem_u32(&ofull[0]), smem_u32(&oempty[0]),
                                    osub, rgs[NS - 1].x, rgs[NS - 1].y, cring_s + Slot::kBorder,
                                    Slot::kBytes, cfull_s, smem_u32(&lempty[0]), lout, lsub,
                                    below.x, crank);
                else
                    run_writer<kSlots>(p, kCl ? g / (int)cn : g, lane, ringo, smem_u32(&ofull[0]), smem_u32(&oempty[0]), osub,
                               rgs[NS - 1].x, rgs[NS - 1].y);
            }
        }
        // ring uses of this group, in blocks of 8 columns
#pragma unroll
        for (int q = 0; q < NS; ++q) csub[q] += (unsigned)(rgs[q].y - rgs[q].x);
        if (gr.writer) osub += (unsigned)(rgs[NS - 1].y - rgs[NS - 1].x);
        auto pages = [](int uses) { return (unsigned)((max(uses, 0) + kLinkPage - 1) / kLinkPage); };
        if (link_in) lin += pages(above.y - rgs[0].x);
        if (link_out) {
            lsub += (unsigned)(below.y - below.x);
            lout += pages(rgs[NS - 1].y - below.x);
        }
    }
    if constexpr (kCl) cluster_sync_all();  // no peer reaches this CTA's shared memory any more
}

template <int DP, int R, int NS, bool kMany, bool kBF = false, bool kSubseq = false,
          bool kT = false>
cudaError_t launch_t(const DpArgs& a, const DpArgs* many, const int2* queue, int items, int* ticket,
                     int num_sms, cudaStream_t s) {
    constexpr int kThreads = split_threads<DP, NS, kBF>();
    const int smem = NS * SplitSmem<DP, R, NS, kBF, false>::kStripBytes;
    auto* kern = k_dp_split<DP, R, NS, kMany, kBF, kSubseq, kT>;
    static DeviceSlots occupancy;
    int blocks_per_sm = 0;
    const cudaError_t e = blocks_per_sm_once(kern, kThreads, smem, occupancy, &blocks_per_sm);
    if (e != cudaSuccess) return e;
    int grid = blocks_per_sm * num_sms;
    if (grid > items) grid = items;
    kern<<<grid, kThreads, smem, s>>>(a, many, queue, items, ticket);
    return cudaGetLastError();
}

}  // namespace
}  // namespace pardtw

// Band map of the parallel backtrace (see bandmap.cu for the whole scheme):
// the per-band, per-segment propagation of entries.
#pragma once
#include "pardtw_common.cuh"

namespace pardtw {

namespace {

constexpr int kNoPath = -2;
constexpr int kOrigin = -1;
constexpr int kMaxBand = 128;

// The backtrace scratch of one pair (bandmap_scratch_bytes(La, Lb) bytes).
struct BtScratch {
    int2* exits;     // nbands x Lb: entries of each band's last two rows
    int2* exits2;    // n2 x Lb: for band b = nbands-2-2m (m < n2, b >= 2), the entries two
                     // bands up (into band b-2's last two rows) of band b's last two rows
    int2* exits4;    // n4 x Lb: for band b = nbands-2-4m (m < n4, b >= 4), the entries four
                     // bands up (into band b-4's last two rows)
    int2* cross;     // nbands: the path's last cell in each band
    int2* seg;       // nbands x band: each band's piece of the path, descending
    int* count;      // nbands: cells in each piece
    int* end_entry;  // the end cell's entry
    int band, nbands, n2, n4;
};
// Bands of La rows, and how many of them have a two-band and a four-band map.
struct BtBands {
    int nbands, n2, n4;
};
__host__ __device__ inline BtBands bt_bands(int La, int band) {
    BtBands r;
    r.nbands = (La + band - 1) / band;
    r.n2 = r.nbands >= 4 ? (r.nbands - 2) / 2 : 0;
    r.n4 = r.nbands >= 6 ? (r.nbands - 6) / 4 + 1 : 0;
    return r;
}
// Bytes of the scratch with bands of `band` rows.
inline size_t bt_scratch_bytes(int La, int Lb, int band) {
    const BtBands r = bt_bands(La, band);
    return (size_t)(r.nbands + r.n2 + r.n4) * Lb * sizeof(int2)  // exits, exits2, exits4
           + (size_t)r.nbands * (1 + band) * sizeof(int2)        // cross, seg
           + (size_t)(r.nbands + 1) * sizeof(int);               // count, end entry
}
__host__ __device__ inline BtScratch bt_scratch(const BtArgs& a) {
    const int La = a.La, Lb = a.Lb;
    const BtBands n = bt_bands(La, a.band);
    BtScratch r;
    r.band = a.band;
    r.nbands = n.nbands;
    r.n2 = n.n2;
    r.n4 = n.n4;
    char* p = static_cast<char*>(a.scratch);
    r.exits = reinterpret_cast<int2*>(p);
    p += (size_t)r.nbands * Lb * sizeof(int2);
    r.exits2 = reinterpret_cast<int2*>(p);
    p += (size_t)r.n2 * Lb * sizeof(int2);
    r.exits4 = reinterpret_cast<int2*>(p);
    p += (size_t)r.n4 * Lb * sizeof(int2);
    r.cross = reinterpret_cast<int2*>(p);
    p += (size_t)r.nbands * sizeof(int2);
    r.seg = reinterpret_cast<int2*>(p);
    p += (size_t)r.nbands * r.band * sizeof(int2);
    r.count = reinterpret_cast<int*>(p);
    p += (size_t)r.nbands * sizeof(int);
    r.end_entry = reinterpret_cast<int*>(p);
    return r;
}


// A segment of a band is mapped by one warp: lane t owns the 32 columns
// s0 + 32 t .. + 31 of the segment's computed range, where s0 = c0 - halo; the
// segment stores columns c0 .. c0 + width - 1 (segments are width apart, the halo
// is twice the band's rows).
//
// Inside a segment an entry is 16 bits, 2 * (column - s0) + (1 if in the band
// above's last row), or one of two codes; a register holds those of columns u
// and u + 8 of a backpointer word, whose fields lie 16 bits apart, so the two
// selects of a cell (bit 1: (1,2), else (2,1); bit 0: (1,1)) are two bitwise
// selects for two cells, by masks that one shift and one byte permute (with sign
// replication) make from the word.  The pairs of columns u-1 and u-2 are the
// registers before; only u = 0, 1 need the neighbouring word (the left lane's by
// two shuffles a row).  What bounds it: these ~108 instructions per row of 1024
// columns, and the loads of the words: four rows at a time (16 bytes), since
// every lane's word lies in a 32-byte sector of its own.  No barriers.  (One
// entry per register, one word per load and a barrier per row of 128 threads
// took 89 us on the 20000 x 25000 pair and 1.5 ms at 100000 x 126231; see
// bandmap.cu for the times now.)
constexpr int kSegCols = 1024;
__host__ __device__ inline int seg_width(int band) { return kSegCols - 2 * band; }
constexpr unsigned kNoPath2 = 0xFFFEFFFEu;  // two columns without a path
constexpr unsigned kOrigin16 = 0xFFFFu;

// 0xFFFF in the half whose field bit (bit 2u + k, and 16 above it) is set: the
// bit shifted to its half's top, then each half filled with the sign of its
// upper byte.
template <int u, int k>
__device__ __forceinline__ unsigned field_mask(unsigned w) {
    unsigned m;
    asm("prmt.b32 %0, %1, %1, 0xBB99;" : "=r"(m) : "r"(w << (15 - 2 * u - k)));
    return m;
}
__device__ __forceinline__ unsigned bit_select(unsigned m, unsigned a, unsigned b) {
    return (m & a) | (~m & b);
}
// The pair left of a word: (high half of l, low half of r).
__device__ __forceinline__ unsigned left_pair(unsigned l, unsigned r) {
    return __byte_perm(l, r, 0x5432u);
}

// Two words' entries of one row: columns u, u + 8 in w[0][u], 16 + u, 24 + u in w[1][u].
struct RowEntries {
    unsigned w[2][8];
};

// Row i from rows i-1 (e1) and i-2 (e2); l1a, l1b, l2a: registers 7 and 6 of the
// left lane's second word in e1 and 7 in e2.
template <int U = 0>
__device__ __forceinline__ void bandmap_pairs(unsigned word, const unsigned* e1, const unsigned* e2,
                                              unsigned q11, unsigned q12, unsigned q21,
                                              unsigned* out) {
    if constexpr (U < 8) {
        // q11 = (column -1, 7), q12 = (-2, 6) of row i-1; q21 = (-1, 7) of row i-2
        const unsigned p11 = U >= 1 ? e1[U >= 1 ? U - 1 : 0] : q11;
        const unsigned p12 = U >= 2 ? e1[U >= 2 ? U - 2 : 0] : (U == 1 ? q11 : q12);
        const unsigned p21 = U >= 1 ? e2[U >= 1 ? U - 1 : 0] : q21;
        const unsigned v = bit_select(field_mask<U, 1>(word), p12, p21);
        out[U] = bit_select(field_mask<U, 0>(word), p11, v);
        bandmap_pairs<U + 1>(word, e1, e2, q11, q12, q21, out);
    }
}

// The band map of band b over segment segx of its columns, by one warp.
template <bool kBanded>
__device__ __forceinline__ void bandmap_segment(const BtArgs& a, int b, int segx, int lane) {
    const uint32_t* __restrict__ bp = a.bp;
    const int La = a.La, Lb = a.Lb, nchunk = a.nchunk, rps = a.rps, wpb = a.wpb;
    const BtScratch sc = bt_scratch(a);
    if (b >= sc.nbands) return;  // warp-uniform, as are the returns below
    const int width = seg_width(sc.band);
    const int r0 = b * sc.band;
    const int r1 = min(r0 + sc.band, La);
    int c0, halo;  // first stored column; columns recomputed to its left (multiple of 16)
    if (kBanded) {
        // segments start at the band's first column over these rows (the
        // ranges are monotone in the strip): every cell left of it has no
        // path, so the first segment needs no halo and the rest of the grid
        // covers only the band's columns
        const int xs = a.ranges[r0 / rps].x * 8, ys = a.ranges[(r1 - 1) / rps].y * 8;
        c0 = (xs & ~(kColsPerWord - 1)) + segx * width;
        if (c0 >= min(ys, Lb)) return;
    } else {
        // Only cells that can lie on a path (path_lo, path_hi): a path
        // cell's predecessors are path cells too, so segments start at
        // path_lo(r0), less the two columns a first step from the band above
        // can come from, (the first without a halo) and end at path_hi(r1-1);
        // the cells left out are never asked for.
        const int xs = max(0, path_lo(r0, La, Lb) - 2);
        const int ys = min(Lb, path_hi(r1 - 1, La, Lb) + 1);
        c0 = (xs & ~(kColsPerWord - 1)) + segx * width;
        if (c0 >= ys) return;
    }
    halo = segx == 0 ? 0 : 2 * sc.band;
    const int s0 = c0 - halo;
    const int jb = s0 + 32 * lane;  // first column of this lane
    // rows r0-2 and r0-1 name themselves: the entries of the cells below them
    RowEntries e1, e2;
#pragma unroll
    for (int h = 0; h < 2; ++h)
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            const unsigned v = 2u * (unsigned)(32 * lane + 16 * h + u);
            const unsigned two = v | ((v + 16u) << 16);
            e1.w[h][u] = b > 0 ? two + 0x00010001u : kNoPath2;
            e2.w[h][u] = b > 0 ? two : kNoPath2;
        }
    // groups of four rows of a strip, 16 bytes a word (a strip's block starts on
    // 16 bytes: wpb is a multiple of 4), loaded two groups ahead
    const int ca = min(jb >> 4, nchunk - 1), cb = min((jb >> 4) + 1, nchunk - 1);
    struct Group {
        uint4 a, b;
        int i, k0, k1;  // row of its first word, words k0 .. k1-1 are rows of the band
    };
    int strip = r0 / rps, lr = r0 - strip * rps, next = r0;  // of the next group to load
    auto load = [&](Group& g) {
        if (next >= r1) {
            g.k0 = g.k1 = 0;
            return;
        }
        const int q = lr >> 2;
        const uint32_t* src = bp + ((size_t)strip * nchunk) * wpb + 4 * q;
        g.a = *reinterpret_cast<const uint4*>(src + (size_t)ca * wpb);
        g.b = *reinterpret_cast<const uint4*>(src + (size_t)cb * wpb);
        g.i = next - (lr & 3);
        g.k0 = lr & 3;
        g.k1 = min(4, min(rps - 4 * q, r1 - g.i));
        next = g.i + g.k1;
        lr = 4 * q + g.k1;
        if (lr >= rps) {
            lr = 0;
            ++strip;
        }
    };
    unsigned l2a = __shfl_up_sync(0xffffffffu, e2.w[1][7], 1);
    if (lane == 0) l2a = kNoPath2;
    auto row = [&](int i, unsigned wa, unsigned wb) {
        unsigned l1a = __shfl_up_sync(0xffffffffu, e1.w[1][7], 1);
        unsigned l1b = __shfl_up_sync(0xffffffffu, e1.w[1][6], 1);
        if (lane == 0) l1a = l1b = kNoPath2;
        RowEntries en;
        bandmap_pairs(wa, e1.w[0], e2.w[0], left_pair(l1a, e1.w[0][7]), left_pair(l1b, e1.w[0][6]),
                      left_pair(l2a, e2.w[0][7]), en.w[0]);
        bandmap_pairs(wb, e1.w[1], e2.w[1], left_pair(e1.w[0][7], e1.w[1][7]),
                      left_pair(e1.w[0][6], e1.w[1][6]), left_pair(e2.w[0][7], e2.w[1][7]),
                      en.w[1]);
        if (kBanded) {
            // cells outside the row's strip range (whole sub-chunks) were never computed
            const int2 rg = __ldg(a.ranges + i / rps);
            const int n0 = jb >> 3;  // the lane's sub-chunks n0 .. n0 + 3
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int n = n0 + 2 * h;
                const unsigned keep = (n >= rg.x && n < rg.y ? 0x0000FFFFu : 0u) |
                                      (n + 1 >= rg.x && n + 1 < rg.y ? 0xFFFF0000u : 0u);
#pragma unroll
                for (int u = 0; u < 8; ++u) en.w[h][u] = bit_select(keep, en.w[h][u], kNoPath2);
            }
        }
        if (i == 0 && jb == 0) en.w[0][0] = (en.w[0][0] & 0xFFFF0000u) | kOrigin16;
        l2a = l1a;
        e2 = e1;
        e1 = en;
    };
    auto rows = [&](const Group& g) {
        const unsigned ga[4] = {g.a.x, g.a.y, g.a.z, g.a.w}, gb[4] = {g.b.x, g.b.y, g.b.z, g.b.w};
        if (g.k0 == 0 && g.k1 == 4) {
#pragma unroll
            for (int k = 0; k < 4; ++k) row(g.i + k, ga[k], gb[k]);
        } else {
#pragma unroll 1
            for (int k = g.k0; k < g.k1; ++k)
                row(g.i + k, k == 0 ? ga[0] : (k == 1 ? ga[1] : (k == 2 ? ga[2] : ga[3])),
                    k == 0 ? gb[0] : (k == 1 ? gb[1] : (k == 2 ? gb[2] : gb[3])));
        }
    };
    Group g0, g1;
    load(g0);
    load(g1);
    while (g0.k1 > 0) {
        const Group g = g0;
        g0 = g1;
        load(g1);
        rows(g);
    }
    auto entry = [&](unsigned v) -> int {  // a 16-bit entry in the column numbers of the matrix
        return v == (kNoPath2 & 0xFFFFu) ? kNoPath : (v == kOrigin16 ? kOrigin : 2 * s0 + (int)v);
    };
    auto half = [&](unsigned pair, int hi) -> unsigned { return hi ? pair >> 16 : pair & 0xFFFFu; };
    if (r1 < La) {
        // the band's last two rows are kept for the band below
        int2* __restrict__ exits = sc.exits + (size_t)b * Lb;
#pragma unroll
        for (int q = 0; q < 32; ++q) {
            const int h = q >> 4, u = q & 7, hi = (q >> 3) & 1;
            const int j = jb + q;
            if (j >= c0 && j < c0 + width && j < Lb)
                exits[j] = make_int2(entry(half(e2.w[h][u], hi)), entry(half(e1.w[h][u], hi)));
        }
    } else {
        // the end cell's entry
        const int q = (Lb - 1) - jb;
        if (q >= 0 && q < 32 && Lb - 1 >= c0 && Lb - 1 < c0 + width) {
#pragma unroll
            for (int v = 0; v < 32; ++v)
                if (v == q) *sc.end_entry = entry(half(e1.w[v >> 4][v & 7], (v >> 3) & 1));
        }
    }
}

}  // namespace
}  // namespace pardtw

// Walking a path back through a backtrace matrix with one warp (the band
// walks of the parallel backtrace, bandmap.cu; the fragment walks of WSDTW,
// wsdtw.cu).  Each step reads one 2-bit field (see step_of_field) whose address
// depends on the step before, so the walk is a chain of loads: from shared
// memory, where the warp first puts every word the next kWalkRows rows can
// need.  From cell (i, j) a path moves at most two columns left per row, so the
// rows i - kWalkRows + 1 .. i of the 17 chunks of 16 columns that end with j's
// hold them (8.7 KB, 68 independent loads a lane).  (With the words in registers
// and neighbouring blocks prefetched from global memory a step took 240 ns and
// the walk of 128 rows 24 us.)
#pragma once
#include "pardtw_common.cuh"

namespace pardtw {
namespace {

constexpr int kWalkRows = 128;
constexpr int kWalkChunks = (2 * (kWalkRows - 1) + 15) / 16 + 1;
constexpr int kWalkWords = kWalkChunks * kWalkRows;

struct WindowWalker {
    const uint32_t* __restrict__ bp;
    int nchunk, rps, wpb, lane;
    uint32_t* sm;   // kWalkWords words of this warp
    int row0, ch1;  // first row and last chunk of the window

    // The window of cell (i, j): all lanes, warp-uniform arguments.
    __device__ __forceinline__ void load(int i, int j) {
        row0 = max(i - kWalkRows + 1, 0);
        ch1 = j >> 4;
        __syncwarp();  // the previous window has been read
        const uint32_t* src[kWalkRows / 32];
#pragma unroll
        for (int m = 0; m < kWalkRows / 32; ++m) {
            const int r = min(row0 + lane + 32 * m, i);
            const int st = r / rps;
            src[m] = bp + ((size_t)st * nchunk) * wpb + (r - st * rps);
        }
#pragma unroll
        for (int k0 = 0; k0 < kWalkChunks; k0 += 6) {
            uint32_t v[6][kWalkRows / 32];
#pragma unroll
            for (int k = 0; k < 6; ++k)
#pragma unroll
                for (int m = 0; m < kWalkRows / 32; ++m)
                    if (k0 + k < kWalkChunks)
                        v[k][m] = __ldg(src[m] + (size_t)max(ch1 - k0 - k, 0) * wpb);
#pragma unroll
            for (int k = 0; k < 6; ++k)
#pragma unroll
                for (int m = 0; m < kWalkRows / 32; ++m)
                    if (k0 + k < kWalkChunks) sm[(k0 + k) * kWalkRows + lane + 32 * m] = v[k][m];
        }
        __syncwarp();
    }
    // A position in the window: r rows below row0, c columns left of its last one.
    __device__ __forceinline__ int row(int i) const { return i - row0; }
    __device__ __forceinline__ int col(int j) const { return 16 * ch1 + 15 - j; }

    // Up to 32 cells of the walk from (r, c), while rows stay at or below rlo and
    // columns in the window and the matrix; returns how many, the first of them in
    // lane 0's (mr, mc), and (r, c) is the cell after the last.  No branch: a walk
    // that has ended stays where it is (a step of a loop with tests and exits took
    // 110 ns).
    __device__ __forceinline__ int steps32(int& r, int& c, int rlo, int& mr, int& mc) const {
        const int climit = min(16 * kWalkChunks, 16 * ch1 + 16);  // columns c of cells
        int n = 0;
#pragma unroll
        for (int u = 0; u < 32; ++u) {
            const bool on = r >= rlo && c < climit;
            if (lane == u) {
                mr = r;
                mc = c;
            }
            const uint32_t w = sm[on ? (c >> 4) * kWalkRows + r : 0];
            const uint32_t f = (w >> (2 * (15 - (c & 15)))) & 3u;
            // moves by field: rows 2, 1, 1, 1, columns 1, 1, 2, 1 (see step_of_field)
            if (on) {
                r -= (0x56 >> (2 * f)) & 3;
                c += (0x65 >> (2 * f)) & 3;
                ++n;
            }
        }
        return n;
    }
};

}  // namespace
}  // namespace pardtw

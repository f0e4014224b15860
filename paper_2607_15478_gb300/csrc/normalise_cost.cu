// Per-frame L2 normalisation and the explicit cosine cost matrix.
//
// The cosine cost of Sec. IV is C[i][j] = 1 - (a_i . b_j) / (|a_i| |b_j|).
// The kernels normalise every frame once (a zero frame stays zero, so its
// cost against anything is 1) and then form 1 - a^_i . b^_j with one FP32
// fused multiply-add per feature, in feature order.  The DP kernel computes
// the cost of each cell the same way on the fly (Sec. II-D: the cost
// matrix is never stored); dtw_cost materialises it for inspection.
#include <cuda_bf16.h>

#include <algorithm>

#include "pardtw_common.cuh"

namespace pardtw {

int padded_dim(int D) {
    static const int sizes[] = {4, 8, 12, 16, 32, 64, 128};
    for (int s : sizes)
        if (D <= s) return s;
    return 0;
}

// kNormFrames frames of A or of B per block.  A is written row-major (La_pad x
// dp), B chunk-transposed (bt_index, Lb_pad frames) or, for the BF16 cost, as
// bf16 rows of kBfStride (Bbf).  Frames of A beyond La, frames of B beyond Lb and
// feature slots beyond D are zero.  The first thread also clears the control
// words of the call.
// Bound by latency and the writes: the block's frames are one stretch of global
// memory, staged as it lies (every load in flight before the first is used), the
// sums of squares run one thread per frame in feature order from shared memory,
// and the results leave in the order of their layout.  (One thread per frame
// reading and writing its own row: 53 us for 51012 frames of D = 100, 5 now; one warp
// per frame for the bf16 rows of 48000 x 128: 120 us.)
constexpr int kNormFrames = 64;
constexpr int kNormThreads = 256;
__host__ __device__ inline int norm_blocks(int La_pad, int Lb_pad) {
    return (La_pad + kNormFrames - 1) / kNormFrames + (Lb_pad + kNormFrames - 1) / kNormFrames;
}

__device__ __forceinline__ void normalise_block(int blk, const NormArgs& a, int D, int dp,
                                                __nv_bfloat16* __restrict__ Bbf) {
    extern __shared__ float sm[];  // kNormFrames rows of D + 1 floats (odd or even: read in order
                                   // of d by one thread per row), then the reciprocal norms
    const int tid = threadIdx.x;
    if (blk == 0 && tid == 0) {
        a.ctl->status = 0;
        a.ctl->detail = 0;
        a.ctl->ticket = 0;
    }
    const int na = (a.La_pad + kNormFrames - 1) / kNormFrames;
    const bool is_a = blk < na;
    const int f0 = (is_a ? blk : blk - na) * kNormFrames;
    const int L = is_a ? a.La : a.Lb, Lp = is_a ? a.La_pad : a.Lb_pad;
    if (f0 >= Lp) return;  // CTA-uniform
    const int S = D | 1;                                    // row stride: conflict-free
    const int have = max(min(kNormFrames, L - f0), 0);      // frames that exist
    const int rows = min(kNormFrames, Lp - f0);             // frames to write
    const float* __restrict__ src = (is_a ? a.A : a.B) + (size_t)f0 * D;
    float* rs = sm + kNormFrames * S;
    {
        // element k = frame k / D, feature k % D, advanced without divisions
        int f = tid / D, d = tid - f * D;
        const int df = kNormThreads / D, dd = kNormThreads - df * D;
        const int n = have * D;
#pragma unroll 8
        for (int k = tid; k < n; k += kNormThreads) {
            sm[f * S + d] = __ldg(src + k);
            f += df;
            d += dd;
            if (d >= D) {
                d -= D;
                ++f;
            }
        }
    }
    __syncthreads();
    if (tid < kNormFrames) {
        float ss = 0.f;
        if (tid < have) {
#pragma unroll 4
            for (int d = 0; d < D; ++d) {
                const float v = sm[tid * S + d];
                ss = fmaf(v, v, ss);
            }
        }
        rs[tid] = ss > 0.f ? 1.0f / sqrtf(ss) : 0.f;
    }
    __syncthreads();
    auto value = [&](int f, int d) { return (f < have && d < D) ? sm[f * S + d] * rs[f] : 0.f; };
    if (is_a) {
        float* __restrict__ out = a.Ahat + (size_t)f0 * dp;
        int f = tid / dp, d = tid - f * dp;
        const int df = kNormThreads / dp, dd = kNormThreads - df * dp;
        for (int k = tid; k < rows * dp; k += kNormThreads) {
            out[k] = value(f, d);
            f += df;
            d += dd;
            if (d >= dp) {
                d -= dp;
                ++f;
            }
        }
    } else if (Bbf) {
        __nv_bfloat16* __restrict__ out = Bbf + (size_t)f0 * kBfStride;
        for (int k = tid; k < rows * kBfStride; k += kNormThreads) {
            const int f = k / kBfStride;
            out[k] = __float2bfloat16_rn(value(f, k - f * kBfStride));
        }
    } else {
        // chunk c, feature d, frame 16 c + e at (c dp + d) 16 + e (bt_index)
        float* __restrict__ out = a.Bt + (size_t)f0 * dp;
        const int e = tid & 15;
        int c = 0, d = tid >> 4;
        for (int k = tid; k < rows * dp; k += kNormThreads) {
            while (d >= dp) {
                d -= dp;
                ++c;
            }
            out[k] = value(16 * c + e, d);
            d += kNormThreads / 16;
        }
    }
}

__global__ void __launch_bounds__(kNormThreads)
    k_normalise(const NormArgs a, int D, int dp, __nv_bfloat16* __restrict__ Bbf) {
    chain_next();
    normalise_block(blockIdx.x, a, D, dp, Bbf);
}

// One pair per blockIdx.y (the grid covers the largest pair); also clears the
// batch's work-queue ticket.
__global__ void __launch_bounds__(kNormThreads)
    k_normalise_many(const NormArgs* __restrict__ many, int D, int dp, int* ticket) {
    const NormArgs a = many[blockIdx.y];
    if (blockIdx.x == 0 && blockIdx.y == 0 && threadIdx.x == 0) *ticket = 0;
    if ((int)blockIdx.x < norm_blocks(a.La_pad, a.Lb_pad))
        normalise_block(blockIdx.x, a, D, dp, nullptr);
}
int norm_smem(int D) { return (kNormFrames * (D | 1) + kNormFrames) * (int)sizeof(float); }

// A replayed batch graph starts with this: a new tag for the border entries
// of every pair (entries left by the previous replay carry the old one).
__global__ void k_bump_epoch(DpArgs* many, int n) {
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= n) return;
    unsigned e = many[k].epoch + 1u;
    many[k].epoch = e == 0u ? 1u : e;
}

cudaError_t launch_bump_epoch(DpArgs* many, int n, cudaStream_t s) {
    k_bump_epoch<<<(n + 127) / 128, 128, 0, s>>>(many, n);
    return cudaGetLastError();
}

cudaError_t launch_normalise(const NormArgs& a, int D, int dp, void* Bbf, cudaStream_t s) {
    k_normalise<<<norm_blocks(a.La_pad, a.Lb_pad), kNormThreads, norm_smem(D), s>>>(
        a, D, dp, static_cast<__nv_bfloat16*>(Bbf));
    return cudaGetLastError();
}

cudaError_t launch_normalise_many(const NormArgs* many, int n, int max_blocks, int D, int dp,
                                  int* ticket, cudaStream_t s) {
    if (n <= 0) return cudaSuccess;
    k_normalise_many<<<dim3((unsigned)max_blocks, (unsigned)n), kNormThreads, norm_smem(D), s>>>(
        many, D, dp, ticket);
    return cudaGetLastError();
}
int normalise_blocks(int La_pad, int Lb_pad) { return norm_blocks(La_pad, Lb_pad); }

// C[i][j] = 1 - sum_d a^_i[d] b^_j[d], accumulated as fma(-a, b, acc) from 1
// in feature order -- bit-identical to the cost the DP kernel uses.
// Writing the matrix is most of the cost of this kernel (4 bytes a cell against
// (La + Lb) * D * 4 bytes read), so it is laid out for the HBM write: a warp covers
// 128 columns, lane l columns l, l + 32, l + 64, l + 96 of them, so every store of
// a row is 128 neighbouring bytes whatever Lb and C's alignment are (4 neighbouring
// columns a lane needed 16-byte stores, and fell to strided ones where a row
// did not start on 16 bytes); the 8 warps of a block write 4 KB of each row.  a^
// comes as 16-byte broadcast loads; the FMAs are paired (two columns each, each
// rounded once).  Blocks take kRows rows at a time, grid-stride; about 16 of them
// per SM, two resident (more registers, for loads in flight, were worth more than
// more warps).  Measured, the whole call (TB/s written; before / now): 12000 x 15000,
// D = 12, 4.06 / 5.7; 11999 x 14999 2.7 / 5.5; D = 16 2.9 / 4.3; D = 20 1.4 / 2.0; 6001 x
// 7003, D = 64, 0.55 / 0.95 (a plain write of such a buffer: 7.3).
constexpr int kCostWarps = 8, kCostCols = 128 * kCostWarps, kCostMaxDp = 128;

// DP <= 16: the lane's 4 columns of b^ stay in registers over all its rows.
// Other widths (DP = 0) load b^ per tile of rows (L1 hits).
template <int DP, int kRows>
__global__ void __launch_bounds__(32 * kCostWarps, 2)
    k_cost(const float* __restrict__ Ahat, int La, const float* __restrict__ Bt, int Lb, int dp,
           float* __restrict__ C) {
    const int lane = threadIdx.x & 31;
    const int jw = blockIdx.x * kCostCols + 128 * (threadIdx.x >> 5);  // the warp's first column
    if (jw >= Lb) return;
    if (DP > 0) dp = DP;
    const float* bcol[4];  // feature d of column c at bcol[c] + 16 d
#pragma unroll
    for (int c = 0; c < 4; ++c) bcol[c] = Bt + bt_index(min(jw + lane + 32 * c, Lb - 1), 0, dp);
    constexpr int kRegD = DP > 0 ? DP : 1;
    float2 b[kRegD][2];
    if constexpr (DP > 0) {
#pragma unroll
        for (int d = 0; d < DP; ++d) {
            b[d][0] = make_float2(__ldg(bcol[0] + 16 * d), __ldg(bcol[1] + 16 * d));
            b[d][1] = make_float2(__ldg(bcol[2] + 16 * d), __ldg(bcol[3] + 16 * d));
        }
    }
    const bool whole = jw + 128 <= Lb;
    for (int i0 = blockIdx.y * kRows; i0 < La; i0 += gridDim.y * kRows) {
        float2 acc[kRows][2];
#pragma unroll
        for (int r = 0; r < kRows; ++r) acc[r][0] = acc[r][1] = make_float2(1.0f, 1.0f);
        // features d0 .. d0 + 3 of the rows (those beyond La read row La - 1 and are
        // never stored)
        auto features = [&](int d0, const float2 (*bb)[2]) {
#pragma unroll
            for (int r = 0; r < kRows; ++r) {
                const float4 a = __ldg(reinterpret_cast<const float4*>(
                    Ahat + (size_t)min(i0 + r, La - 1) * dp + d0));
                const float av[4] = {a.x, a.y, a.z, a.w};
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    const float2 x = make_float2(-av[u], -av[u]);
                    acc[r][0] = __ffma2_rn(x, bb[u][0], acc[r][0]);
                    acc[r][1] = __ffma2_rn(x, bb[u][1], acc[r][1]);
                }
            }
        };
        if constexpr (DP > 0) {
#pragma unroll
            for (int d0 = 0; d0 < DP; d0 += 4) features(d0, b + d0);
        } else {
            for (int d0 = 0; d0 < dp; d0 += 4) {
                float2 t[4][2];
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    t[u][0] = make_float2(__ldg(bcol[0] + 16 * (d0 + u)), __ldg(bcol[1] + 16 * (d0 + u)));
                    t[u][1] = make_float2(__ldg(bcol[2] + 16 * (d0 + u)), __ldg(bcol[3] + 16 * (d0 + u)));
                }
                features(d0, t);
            }
        }
        float* out = C + (size_t)i0 * Lb + jw + lane;
        if (whole && i0 + kRows <= La) {
#pragma unroll
            for (int r = 0; r < kRows; ++r, out += Lb) {
                __stcs(out, acc[r][0].x);
                __stcs(out + 32, acc[r][0].y);
                __stcs(out + 64, acc[r][1].x);
                __stcs(out + 96, acc[r][1].y);
            }
        } else {
#pragma unroll
            for (int r = 0; r < kRows; ++r, out += Lb) {
                const float v[4] = {acc[r][0].x, acc[r][0].y, acc[r][1].x, acc[r][1].y};
#pragma unroll
                for (int c = 0; c < 4; ++c)
                    if (i0 + r < La && jw + lane + 32 * c < Lb) __stcs(out + 32 * c, v[c]);
            }
        }
    }
}

cudaError_t launch_cost(const float* Ahat, int La, const float* Bt, int Lb, int dp, float* C,
                        cudaStream_t s) {
    if (dp > kCostMaxDp || dp % 4 != 0) return cudaErrorInvalidValue;
    constexpr int kFew = 4, kMany = 8;  // rows a tile with b^ in registers, with b^ loaded per tile
    const int rows = dp <= 16 ? kFew : kMany;
    const int gx = (Lb + kCostCols - 1) / kCostCols;
    const int ty = (La + rows - 1) / rows;
    const int gy = std::min(std::min((2432 + gx - 1) / gx, ty), 65535);
    const dim3 grid((unsigned)gx, (unsigned)gy);
    const int threads = 32 * kCostWarps;
    switch (dp) {
        case 4: k_cost<4, kFew><<<grid, threads, 0, s>>>(Ahat, La, Bt, Lb, dp, C); break;
        case 8: k_cost<8, kFew><<<grid, threads, 0, s>>>(Ahat, La, Bt, Lb, dp, C); break;
        case 12: k_cost<12, kFew><<<grid, threads, 0, s>>>(Ahat, La, Bt, Lb, dp, C); break;
        case 16: k_cost<16, kFew><<<grid, threads, 0, s>>>(Ahat, La, Bt, Lb, dp, C); break;
        default: k_cost<0, kMany><<<grid, threads, 0, s>>>(Ahat, La, Bt, Lb, dp, C); break;
    }
    return cudaGetLastError();
}

}  // namespace pardtw

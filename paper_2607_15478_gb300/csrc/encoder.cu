// Band encoder of the learned band (dtw_align_learned): a small 1-D
// convolutional network over the sequences averaged over `ds` frames.  The
// paper only names bands and multiscale DTW as ways to cut the quadratic cost
// (Sec. II); the network, its loss and its use are this library's.
//
//   x      = pooled frames (mean of ds frames), L2-normalised   [Lc][D]
//   h1     = relu(conv5(x,  W1) + b1)                            [Lc][64]
//   h2     = relu(conv5(h1, W2) + b2)                            [Lc][64]
//   h3     = relu(conv5(h2, W3) + b3)                            [Lc][64]
//   z      = W4 h3 + b4,  e = z / |z|  (the embedding)           [Lc][16]
//   s      = W5 . h3 + b5 (half-width logit; rows of A only)     [Lc]
//   halfwidth = wmin * (wmax / wmin)^sigmoid(s)   in fine frames
//
// conv5 is a 1-D convolution of width 5 with zero padding 2:
//   y[l][co] = sum_{ci, t} W[co][ci][t] x[l + t - 2][ci].
// The coarse alignment is the exact DTW of eA against eB (cosine cost), and
// the band around its upsampled path has the predicted half-width.
//
// Training (dtw_encoder_grad): mode 0 is a contrastive loss on the
// embeddings, for each coarse row i of A a softmax over the coarse columns
// within kWin of the column c_i that the exact path matches to the row,
// loss_i = -log softmax_j(eA_i . eB_j / tau)[c_i]; mode 1 fits the width head
// (trunk frozen) with a pinball loss at quantile kQ to the half-width the
// band of the coarse path needs to hold the exact path.  Gradients are the
// hand-derived backward passes of the layers above (no autodiff), summed into
// the caller's gradient array with atomics.
//
// Kernels: k_pool_norm, k_conv (forward, and backward-data with transposed
// flipped weights), k_conv_wgrad, k_embed, k_embed_bwd, k_head_grad (the head
// weights' gradients), k_targets, k_loss_emb, k_width_target, k_loss_width,
// k_adam.  The layers of both sequences run in one launch each (EncRows2:
// blockIdx.z is the sequence): a coarse sequence of a training pair has one to
// three thousand rows, so a launch of its own and tiles of 64 rows and 64
// channels left most SMs idle (a training step of 12000 x 14500 frames took 1.31 ms
// that way, 0.84 of it in k_conv_wgrad on 12 of the 152 SMs; 0.14 ms now).
#include "pardtw_common.cuh"

#include <cuda_bf16.h>

namespace pardtw {

namespace {

constexpr int kC = kEncChannels;   // 64
constexpr int kE = kEncEmbed;      // 16
constexpr int kK = kEncKernel;     // 5
constexpr int kPad = kK / 2;
constexpr int kWin = 16;           // contrastive window half-width (coarse columns)
constexpr float kTau = 0.1f;       // softmax temperature
constexpr float kQ = 0.9f;         // pinball quantile of the width loss
constexpr float kMargin = 64.0f;   // fine frames added to the needed half-width

__device__ __forceinline__ float round_bf16(float x) {
    return __bfloat162float(__float2bfloat16_rn(x));
}

// Mean of each window of ds frames (the last may be shorter), L2-normalised
// (a zero mean stays zero).  kG lanes per pooled frame, one (two for D > 32)
// feature(s) a lane; the sum of squares runs over the features in order.
template <int kG>
__global__ void __launch_bounds__(128) k_pool_norm(const EncRows2 q, int D, int ds) {
    const EncRows a = blockIdx.z ? q.s[1] : q.s[0];
    const int L = a.L, Lc = (L + ds - 1) / ds;
    const int c = (blockIdx.x * blockDim.x + threadIdx.x) / kG;
    const int g = threadIdx.x % kG;
    const int f0 = min(c, Lc - 1) * ds, f1 = min(f0 + ds, L);
    float v[2] = {0.f, 0.f};
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const int d = g + h * kG;
        if (d < D) {
            float acc = 0.f;
#pragma unroll 8
            for (int f = f0; f < f1; ++f) acc += __ldg(a.X + (size_t)f * D + d);
            v[h] = acc / (float)(f1 - f0);
        }
    }
    float ss = 0.f;
    for (int d = 0; d < D; ++d) {
        const float x = __shfl_sync(0xffffffffu, d < kG ? v[0] : v[1], d % kG, kG);
        ss = fmaf(x, x, ss);
    }
    const float r = ss > 0.f ? rsqrtf(ss) : 0.f;
    if (c >= Lc) return;
#pragma unroll
    for (int h = 0; h < 2; ++h)
        if (g + h * kG < D) a.Y[(size_t)c * D + g + h * kG] = v[h] * r;
}

// Generic conv5 over kTL rows and kCO output channels per block:
//   Y[l][co] = bias[co] + sum_{ci < Cin, t} Wt(ci, t, co) * Xm[l + t - 2][ci]
// Xm = X masked by (mask > 0) where mask is given (the relu derivative of
// the layer whose gradient X is).  Wt(ci, t, co) = W[co][ci][t] (forward,
// W: [kC][Cin][kK]) or, with kBwd, W[ci][co][kK-1-t] (backward data: W is the
// forward weight [Cin_b = kC][Cout_b][kK] read transposed and flipped).
// kBF16: inputs and weights rounded to bf16 (products exact in FP32, FP32
// accumulation).
// Thread t computes rows 4 (t / 8) .. + 3 and channels 2 (t % 8), + 1 of the
// tile, each output by the same FMAs in the same order (input channel outer,
// tap inner) as one thread per output would: per input channel 8 rows of X and
// 5 x 2 weights from shared memory feed 40 FMAs.  A block has a quarter of the
// channels: the weights it stages (20 KB at Cin = 64) are read from global
// memory in order, and 1500 rows make 96 blocks instead of 24 (28 us a layer of
// 1500 rows at Cin = 64 with all 64 channels a block, 10 us for both sequences of
// a pair now; bound by the staging and 64 dependent channel steps of few warps).
constexpr int kTL = 64;
constexpr int kCO = 16;
constexpr int kWS = kCO + 2;         // floats per (ci, t) row of staged weights
constexpr int kConvThreads = 128;
constexpr int kXS = kTL + 2 * kPad;  // rows of X per input channel in shared memory
static_assert(kConvThreads == (kTL / 4) * (kCO / 2), "4 rows x 2 channels a thread");

// kCin: the input channels (64: loads of 16 bytes, all in flight before the
// first is stored), 0: Cin of them, one value at a time.
template <int kCin, bool kBwd, bool kBF16>
__global__ void __launch_bounds__(kConvThreads)
    k_conv(const EncRows2 q, int Cin, const float* __restrict__ W, const float* __restrict__ bias,
           int relu) {
    static_assert(kCin == 0 || kCin == kC, "whole rows of 16-byte words");
    if (kCin > 0) Cin = kCin;
    extern __shared__ __align__(16) float sm[];
    float* Xs = sm;                       // [Cin][kXS]
    float* Ws = sm + Cin * kXS;           // [Cin * kK][kWS]
    const EncRows a = blockIdx.z ? q.s[1] : q.s[0];
    const int L = a.L;
    const int l0 = blockIdx.x * kTL, co0 = blockIdx.y * kCO;
    if (l0 >= L) return;
    const float* __restrict__ X = a.X;
    const float* __restrict__ mask = a.M;
    const int tid = threadIdx.x;
    auto put_w = [&](int k, float w) {  // value k of the block's weights
        int co, ct;
        if (kBwd) {  // per ci, kCO x kK consecutive values
            const int ci = k / (kCO * kK), r = k - ci * (kCO * kK);
            co = r / kK;
            ct = ci * kK + (kK - 1 - (r - co * kK));
        } else {  // per channel, Cin x kK consecutive values
            co = k / (Cin * kK);
            ct = k - co * (Cin * kK);
        }
        Ws[ct * kWS + co] = kBF16 ? round_bf16(w) : w;
    };
    auto w_index = [&](int k) -> size_t {
        if (!kBwd) return (size_t)co0 * Cin * kK + k;
        const int ci = k / (kCO * kK);
        return ((size_t)ci * kC + co0) * kK + (k - ci * (kCO * kK));
    };
    auto put_x = [&](int r, int ci, float v) { Xs[ci * kXS + r] = kBF16 ? round_bf16(v) : v; };
    if constexpr (kCin > 0) {
        constexpr int kWV = kCin * kK * kCO / 4, kXV = kXS * kCin / 4;
        constexpr int kNW = kWV / kConvThreads, kNX = (kXV + kConvThreads - 1) / kConvThreads;
        static_assert(kWV % kConvThreads == 0, "whole batches of weights");
        float4 w[kNW], x[kNX];
#pragma unroll
        for (int u = 0; u < kNW; ++u) {
            const float* src = W + w_index(4 * (tid + u * kConvThreads));
            // a segment starts on a 16-byte boundary only where W does
            w[u] = make_float4(__ldg(src), __ldg(src + 1), __ldg(src + 2), __ldg(src + 3));
        }
#pragma unroll
        for (int u = 0; u < kNX; ++u) {
            const int k = tid + u * kConvThreads;
            const int l = l0 + k / (kCin / 4) - kPad;
            x[u] = make_float4(0.f, 0.f, 0.f, 0.f);
            if (k < kXV && l >= 0 && l < L) {
                const size_t o = (size_t)l * (kCin / 4) + k % (kCin / 4);
                x[u] = __ldg(reinterpret_cast<const float4*>(X) + o);
                if (kBwd && mask) {
                    const float4 m = __ldg(reinterpret_cast<const float4*>(mask) + o);
                    if (!(m.x > 0.f)) x[u].x = 0.f;
                    if (!(m.y > 0.f)) x[u].y = 0.f;
                    if (!(m.z > 0.f)) x[u].z = 0.f;
                    if (!(m.w > 0.f)) x[u].w = 0.f;
                }
            }
        }
#pragma unroll
        for (int u = 0; u < kNW; ++u) {
            const int k = 4 * (tid + u * kConvThreads);
            put_w(k, w[u].x);
            put_w(k + 1, w[u].y);
            put_w(k + 2, w[u].z);
            put_w(k + 3, w[u].w);
        }
#pragma unroll
        for (int u = 0; u < kNX; ++u) {
            const int k = tid + u * kConvThreads;
            if (k < kXV) {
                const int r = k / (kCin / 4), ci = 4 * (k % (kCin / 4));
                put_x(r, ci, x[u].x);
                put_x(r, ci + 1, x[u].y);
                put_x(r, ci + 2, x[u].z);
                put_x(r, ci + 3, x[u].w);
            }
        }
    } else {
        for (int k = tid; k < Cin * kK * kCO; k += kConvThreads) put_w(k, W[w_index(k)]);
        for (int k = tid; k < kXS * Cin; k += kConvThreads) {
            const int r = k / Cin, ci = k % Cin;
            const int l = l0 + r - kPad;
            float v = 0.f;
            if (l >= 0 && l < L) {
                v = X[(size_t)l * Cin + ci];
                if (mask && !(mask[(size_t)l * Cin + ci] > 0.f)) v = 0.f;
            }
            put_x(r, ci, v);
        }
    }
    __syncthreads();
    const int cg = tid % (kCO / 2), rg = tid / (kCO / 2);  // channels 2 cg, +1, rows 4 rg ..
    float acc[4][2];
#pragma unroll
    for (int i = 0; i < 4; ++i) acc[i][0] = acc[i][1] = 0.f;
#pragma unroll 4
    for (int ci = 0; ci < Cin; ++ci) {
        // rows 4 rg .. 4 rg + 7 of the tile (with the halo): the taps' inputs
        const float4 xa = *reinterpret_cast<const float4*>(Xs + ci * kXS + 4 * rg);
        const float4 xb = *reinterpret_cast<const float4*>(Xs + ci * kXS + 4 * rg + 4);
        const float x[8] = {xa.x, xa.y, xa.z, xa.w, xb.x, xb.y, xb.z, xb.w};
#pragma unroll
        for (int t = 0; t < kK; ++t) {
            const float2 w = *reinterpret_cast<const float2*>(Ws + (ci * kK + t) * kWS + 2 * cg);
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                acc[i][0] = fmaf(w.x, x[i + t], acc[i][0]);
                acc[i][1] = fmaf(w.y, x[i + t], acc[i][1]);
            }
        }
    }
    const int co = co0 + 2 * cg;
    const float b0 = bias ? bias[co] : 0.f, b1 = bias ? bias[co + 1] : 0.f;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const int l = l0 + 4 * rg + i;
        if (l < L) {
            float y0 = acc[i][0] + b0, y1 = acc[i][1] + b1;
            if (relu) {
                y0 = fmaxf(y0, 0.f);
                y1 = fmaxf(y1, 0.f);
            }
            *reinterpret_cast<float2*>(a.Y + (size_t)l * kC + co) = make_float2(y0, y1);
        }
    }
}

// Weight gradient of a conv5 layer over a tile of kTW rows and kCI input
// channels:
//   dW[co][ci][t] += sum_l dYm[l][co] X[l + t - 2][ci],  db[co] += sum_l dYm[l][co]
// dYm = dY masked by (Yout > 0) (the layer's relu).  Thread (co, cg) owns two
// input channels for all t, whose rows it keeps in a sliding window.  (128 rows
// and every input channel a block left 12 blocks on 1500 rows: 210 us a layer at
// Cin = 64.)  Bound by the atomics of its sums: 20 us a layer for both sequences
// of a pair with one tile a block, a training step 152, 140, 146, 145 us with 1, 2,
// 3, 4 tiles.
constexpr int kTW = 64;     // rows staged at a time
constexpr int kTiles = 2;   // of which a block takes so many: its sums go out by atomics once
constexpr int kCI = 8;
constexpr int kWgThreads = kC * (kCI / 2);
__global__ void __launch_bounds__(kWgThreads)
    k_conv_wgrad(const EncGrad2 q, int Cin, float* __restrict__ dW, float* __restrict__ db) {
    __shared__ __align__(16) float Gs[kTW][kC];
    __shared__ __align__(8) float Xs[kTW + 2 * kPad][kCI];
    const EncGrad a = blockIdx.z ? q.s[1] : q.s[0];
    const int L = a.L;
    const int l0b = blockIdx.x * (kTW * kTiles), ci0 = blockIdx.y * kCI;
    if (l0b >= L) return;
    const int tid = threadIdx.x;
    const int co = tid % kC, cg = tid / kC;
    float acc[2][kK];
    float bacc = 0.f;
#pragma unroll
    for (int t = 0; t < kK; ++t) acc[0][t] = acc[1][t] = 0.f;
    for (int l0 = l0b; l0 < min(l0b + kTW * kTiles, L); l0 += kTW) {
        __syncthreads();  // the previous tile has been read
        constexpr int kNG = kTW * kC / 4 / kWgThreads;  // 16-byte words per thread
        float4 gv[kNG], yv[kNG];
#pragma unroll
        for (int u = 0; u < kNG; ++u) {
            const int k = tid + u * kWgThreads;
            const int l = l0 + k / (kC / 4);
            gv[u] = yv[u] = make_float4(0.f, 0.f, 0.f, 0.f);
            if (l < L) {
                const size_t o = (size_t)l * (kC / 4) + k % (kC / 4);
                gv[u] = __ldg(reinterpret_cast<const float4*>(a.dY) + o);
                yv[u] = __ldg(reinterpret_cast<const float4*>(a.Yout) + o);
            }
        }
#pragma unroll
        for (int u = 0; u < kNG; ++u) {
            const int k = tid + u * kWgThreads;
            *reinterpret_cast<float4*>(&Gs[k / (kC / 4)][4 * (k % (kC / 4))]) =
                make_float4(yv[u].x > 0.f ? gv[u].x : 0.f, yv[u].y > 0.f ? gv[u].y : 0.f,
                            yv[u].z > 0.f ? gv[u].z : 0.f, yv[u].w > 0.f ? gv[u].w : 0.f);
        }
#pragma unroll
        for (int k = tid; k < (kTW + 2 * kPad) * kCI; k += kWgThreads) {
            const int r = k / kCI, ci = ci0 + k % kCI;
            const int l = l0 + r - kPad;
            Xs[r][k % kCI] = (l >= 0 && l < L && ci < Cin) ? a.X[(size_t)l * Cin + ci] : 0.f;
        }
        __syncthreads();
        constexpr int kU = 8;
        float2 x[kU + 2 * kPad];  // rows r .. r + kU + 3 of the two channels
#pragma unroll
        for (int t = 0; t < 2 * kPad; ++t) x[t] = *reinterpret_cast<const float2*>(&Xs[t][2 * cg]);
        for (int r = 0; r < kTW; r += kU) {
            float g[kU];
#pragma unroll
            for (int u = 0; u < kU; ++u) {
                x[2 * kPad + u] = *reinterpret_cast<const float2*>(&Xs[r + 2 * kPad + u][2 * cg]);
                g[u] = Gs[r + u][co];
            }
#pragma unroll
            for (int u = 0; u < kU; ++u) {
                bacc += g[u];
#pragma unroll
                for (int t = 0; t < kK; ++t) {
                    acc[0][t] = fmaf(g[u], x[u + t].x, acc[0][t]);
                    acc[1][t] = fmaf(g[u], x[u + t].y, acc[1][t]);
                }
            }
#pragma unroll
            for (int t = 0; t < 2 * kPad; ++t) x[t] = x[kU + t];
        }
    }
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const int ci = ci0 + 2 * cg + h;
        if (ci < Cin)
#pragma unroll
            for (int t = 0; t < kK; ++t) atomicAdd(&dW[((size_t)co * Cin + ci) * kK + t], acc[h][t]);
    }
    if (blockIdx.y == 0 && cg == 0) atomicAdd(&db[co], bacc);
}

// Heads, four threads per row (four embedding components each): z = W4 h3 + b4,
// e = z / |z| (invn = 1/|z|, 0 for z = 0), s = W5 . h3 + b5 and the half-width in
// fine frames.  Sums run over the channels, and the norm over the components,
// in order.  G, jsum, cnt (may be null): zeroed, a training step's embedding gradient and
// the sums of its targets.
__global__ void __launch_bounds__(128) k_embed(const EncEmbed2 q, const float* __restrict__ W4,
                        const float* __restrict__ b4, const float* __restrict__ W5,
                        const float* __restrict__ b5, int bf16, float wmin, float wmax) {
    __shared__ __align__(16) float w4[kC * kE];  // [c][e]
    __shared__ float w5[kC], bb[kE + 1];
    const EncEmbed a = blockIdx.z ? q.s[1] : q.s[0];
    const int L = a.L;
    if (blockIdx.x * 32 >= L) return;
#pragma unroll
    for (int k = threadIdx.x; k < kE * kC; k += 128) {
        const float w = W4[k];
        w4[(k % kC) * kE + k / kC] = bf16 ? round_bf16(w) : w;
    }
    for (int k = threadIdx.x; k < kC; k += blockDim.x) w5[k] = W5[k];
    if (threadIdx.x < kE) bb[threadIdx.x] = b4[threadIdx.x];
    if (threadIdx.x == 0) bb[kE] = b5[0];
    __syncthreads();
    const int l = blockIdx.x * 32 + threadIdx.x / 4, eg = threadIdx.x % 4;
    const int lr = min(l, L - 1);  // every lane takes part in the shuffles
    float z[4] = {0.f, 0.f, 0.f, 0.f};
    float s = 0.f;
    const float4* h4 = reinterpret_cast<const float4*>(a.H + (size_t)lr * kC);
#pragma unroll 4
    for (int c4 = 0; c4 < kC / 4; ++c4) {
        const float4 v = h4[c4];
        const float hv[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int c = 4 * c4 + u;
            const float hc = bf16 ? round_bf16(hv[u]) : hv[u];
            const float4 w = *reinterpret_cast<const float4*>(w4 + c * kE + 4 * eg);
            z[0] = fmaf(w.x, hc, z[0]);
            z[1] = fmaf(w.y, hc, z[1]);
            z[2] = fmaf(w.z, hc, z[2]);
            z[3] = fmaf(w.w, hc, z[3]);
            s = fmaf(w5[c], hv[u], s);
        }
    }
    float ss = 0.f;
#pragma unroll
    for (int k = 0; k < 4; ++k) z[k] += bb[4 * eg + k];
#pragma unroll
    for (int step = 0; step < 4; ++step) {
        float mine = ss;
#pragma unroll
        for (int k = 0; k < 4; ++k) mine = fmaf(z[k], z[k], mine);
        ss = __shfl_sync(0xffffffffu, mine, step, 4);
    }
    const float r = ss > 0.f ? rsqrtf(ss) : 0.f;
    if (l >= L) return;
    reinterpret_cast<float4*>(a.Emb + (size_t)l * kE)[eg] =
        make_float4(z[0] * r, z[1] * r, z[2] * r, z[3] * r);
    if (a.G) reinterpret_cast<float4*>(a.G + (size_t)l * kE)[eg] = make_float4(0.f, 0.f, 0.f, 0.f);
    if (eg != 0) return;
    if (a.jsum) {
        a.jsum[l] = 0ull;
        a.cnt[l] = 0;
    }
    if (a.invn) a.invn[l] = r;
    s += bb[kE];
    if (a.S) a.S[l] = s;
    if (a.HW) {
        const float sg = 1.f / (1.f + expf(-s));
        a.HW[l] = wmin * exp2f(sg * log2f(wmax / wmin));
    }
}

// Backward of the embedding head, kBwdRows rows per block: ge = dL/de -> dz =
// (ge - e (e.ge)) * invn, stored in place of ge; dH[l][c] = sum_e W4[e][c] dz[e].
// Thread (row slot, c): a row's 64 channels are written side by side.
constexpr int kBwdRows = 16;
__global__ void __launch_bounds__(256) k_embed_bwd(const EncEmbed2 q, const float* __restrict__ W4) {
    __shared__ float w4[kE * kC];
    __shared__ float es[kBwdRows][kE], gs[kBwdRows][kE];
    const EncEmbed a = blockIdx.z ? q.s[1] : q.s[0];
    const int L = a.L;
    const int l0 = blockIdx.x * kBwdRows;
    if (l0 >= L) return;
    for (int k = threadIdx.x; k < kE * kC; k += blockDim.x) w4[k] = W4[k];
    const int r = threadIdx.x / kE, k = threadIdx.x % kE;  // 16 rows x 16 components
    const int l = l0 + r;
    if (l < L) {
        es[r][k] = a.Emb[(size_t)l * kE + k];
        gs[r][k] = a.G[(size_t)l * kE + k];
    }
    __syncthreads();
    float dz = 0.f;
    if (l < L) {
        float dot = 0.f;
#pragma unroll
        for (int e = 0; e < kE; ++e) dot = fmaf(es[r][e], gs[r][e], dot);
        dz = (gs[r][k] - es[r][k] * dot) * a.invn[l];
        a.G[(size_t)l * kE + k] = dz;
    }
    __syncthreads();
    gs[r][k] = dz;
    __syncthreads();
    const int c = threadIdx.x % kC;
    for (int row = threadIdx.x / kC; row < kBwdRows && l0 + row < L; row += 256 / kC) {
        float acc = 0.f;
#pragma unroll
        for (int e = 0; e < kE; ++e) acc = fmaf(w4[e * kC + c], gs[row][e], acc);
        a.dH[(size_t)(l0 + row) * kC + c] = acc;
    }
}

// Gradients of a head over a tile of kHeadRows rows: dWh[e][c] += sum_l U[l][e]
// H[l][c], dbh[e] += sum_l U[l][e], for kN = 16 (embedding) or 1 (half-width)
// outputs.  Thread (c, eg) owns channel c of kN / 4 (or all) outputs.
constexpr int kHeadRows = 32;
template <int kN>
__global__ void __launch_bounds__(256) k_head_grad(const EncHead2 q, float* __restrict__ dWh,
                                                   float* __restrict__ dbh) {
    constexpr int kPer = kN >= 4 ? kN / 4 : 1;
    __shared__ __align__(16) float us[kHeadRows][kN];
    const EncHead a = blockIdx.z ? q.s[1] : q.s[0];
    const int l0 = blockIdx.x * kHeadRows;
    if (l0 >= a.L) return;
    const int n = min(kHeadRows, a.L - l0);
    for (int k = threadIdx.x; k < n * kN; k += blockDim.x) us[k / kN][k % kN] = a.U[(size_t)l0 * kN + k];
    __syncthreads();
    const int c = threadIdx.x % kC, eg = threadIdx.x / kC;
    if (kPer * eg >= kN) return;
    float acc[kPer], bacc[kPer];
#pragma unroll
    for (int k = 0; k < kPer; ++k) acc[k] = bacc[k] = 0.f;
#pragma unroll 8
    for (int r = 0; r < n; ++r) {
        const float h = a.H[(size_t)(l0 + r) * kC + c];
#pragma unroll
        for (int k = 0; k < kPer; ++k) {
            const float u = us[r][kPer * eg + k];
            acc[k] = fmaf(u, h, acc[k]);
            bacc[k] += u;
        }
    }
#pragma unroll
    for (int k = 0; k < kPer; ++k) {
        atomicAdd(&dWh[(kPer * eg + k) * kC + c], acc[k]);
        if (c == 0) atomicAdd(&dbh[kPer * eg + k], bacc[k]);
    }
}

// First of the n path entries whose row is >= row (rows ascend along a path).
__device__ __forceinline__ int first_of_row(const int32_t* __restrict__ path, int n, int row) {
    int lo = 0, hi = n;
    while (lo < hi) {
        const int mid = (lo + hi) >> 1;
        if (path[2 * mid] < row)
            lo = mid + 1;
        else
            hi = mid;
    }
    return lo;
}

// Coarse column matched to every coarse row of A by the exact fine path:
// the mean column of the path entries in the row's ds fine rows, divided by
// ds.  One thread per path entry, in whatever order they come, adds to its row's
// sum and count (zeroed by k_embed); k_loss_emb divides.
__global__ void k_targets(const int32_t* __restrict__ path, const int* __restrict__ plen, int cap,
                          int ds, int Lac, unsigned long long* __restrict__ jsum,
                          int* __restrict__ cnt) {
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= min(*plen, cap)) return;
    const int2 c = make_int2(path[2 * k], path[2 * k + 1]);
    const int i = c.x / ds;
    if (c.x < 0 || i >= Lac) return;
    atomicAdd(&jsum[i], (unsigned long long)c.y);
    atomicAdd(&cnt[i], 1);
}
__device__ __forceinline__ int target_column(unsigned long long jsum, int n, int ds, int Lbc) {
    // every fine row lies on a path except rows a (2,1) step skips; a coarse
    // row of ds >= 2 fine rows always holds one
    if (n == 0) return min(0, Lbc - 1);
    // (the same whole number in 32 bits: below 2^52 no rounding reaches the next one)
    const unsigned long long rows = (unsigned long long)n * (unsigned)ds;
    if (((jsum | rows) >> 32) == 0) return min((int)((unsigned)jsum / (unsigned)rows), Lbc - 1);
    const double m = (double)jsum / n;
    return min((int)(m / ds), Lbc - 1);
}

// Contrastive loss, one warp per coarse row i of A (see the file comment),
// lane k at column j0 + k of its window (lane 0 also at j0 + 32).  gA[i] = dL/deA_i
// is written; dL/deB_j is added to gB with atomics, 16 neighbouring floats at a
// time.  The loss is the mean over rows.  (One thread per row took 75 us on 1500
// rows: 528 atomics and three passes over its window each.)
constexpr int kLossRows = 4;
__global__ void __launch_bounds__(32 * kLossRows)
    k_loss_emb(const float* __restrict__ eA, int Lac, const float* __restrict__ eB, int Lbc,
               const unsigned long long* __restrict__ jsum, const int* __restrict__ cnt, int ds,
               float* __restrict__ gA, float* __restrict__ gB, float* __restrict__ loss) {
    constexpr int kWidth = 2 * kWin + 1;
    static_assert(kWidth == 33, "a lane per column and one more");
    __shared__ float s_w[kLossRows][kWidth], s_a[kLossRows][kE], s_loss[kLossRows];
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int i = blockIdx.x * kLossRows + w;
    float row_loss = 0.f;
    const float inv_n = 1.f / (float)Lac;
    if (i < Lac) {
        if (lane < kE) s_a[w][lane] = eA[(size_t)i * kE + lane];
        __syncwarp();
        const int c = target_column(jsum[i], cnt[i], ds, Lbc);
        const int j0 = max(c - kWin, 0), j1 = min(c + kWin, Lbc - 1);
        float lg[2] = {-INFINITY, -INFINITY};
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int j = j0 + lane + 32 * h;
            if (j <= j1) {
                const float4* b = reinterpret_cast<const float4*>(eB + (size_t)j * kE);
                float d = 0.f;
#pragma unroll
                for (int e4 = 0; e4 < kE / 4; ++e4) {
                    const float4 v = b[e4];
                    d = fmaf(s_a[w][4 * e4], v.x, d);
                    d = fmaf(s_a[w][4 * e4 + 1], v.y, d);
                    d = fmaf(s_a[w][4 * e4 + 2], v.z, d);
                    d = fmaf(s_a[w][4 * e4 + 3], v.w, d);
                }
                lg[h] = d / kTau;
            }
        }
        float mx = fmaxf(lg[0], lg[1]);
#pragma unroll
        for (int off = 16; off > 0; off >>= 1)
            mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, off));
        float se = 0.f;
#pragma unroll
        for (int h = 0; h < 2; ++h)
            if (j0 + lane + 32 * h <= j1) se += expf(lg[h] - mx);
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) se += __shfl_xor_sync(0xffffffffu, se, off);
        const float lse = mx + logf(se);
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int j = j0 + lane + 32 * h;
            if (j <= j1) {
                const float pj = expf(lg[h] - lse) - (j == c ? 1.f : 0.f);
                s_w[w][lane + 32 * h] = pj * inv_n / kTau;
                if (j == c) s_loss[w] = (lse - lg[h]) * inv_n;
            }
        }
        __syncwarp();
        row_loss = s_loss[w];
        const int n = j1 - j0 + 1;
        // component lane % 16 over the even (lanes 0-15) and odd columns, then both
        const int e = lane % kE;
        float ga = 0.f;
        for (int k = lane / kE; k < n; k += 2)
            ga = fmaf(s_w[w][k], eB[(size_t)(j0 + k) * kE + e], ga);
        ga += __shfl_xor_sync(0xffffffffu, ga, kE);
        if (lane < kE) gA[(size_t)i * kE + e] = ga;
        for (int k = lane; k < n * kE; k += 32)
            atomicAdd(&gB[(size_t)j0 * kE + k], s_w[w][k / kE] * s_a[w][k % kE]);
    }
    __syncthreads();
    if (lane == 0) s_loss[w] = row_loss;
    __syncthreads();
    if (threadIdx.x == 0) {
        float sum = 0.f;
#pragma unroll
        for (int k = 0; k < kLossRows; ++k) sum += s_loss[k];
        atomicAdd(loss, sum);
    }
}

// Width target of every coarse row i of A, in [0, 1] on the log scale of the
// half-width: the band of the coarse path at w = 0 over coarse rows
// i-1 .. i+1 spans fine columns [jmin ds, (jmax + 1) ds - 1]; the row needs
// the distance from that span of the exact path's columns in its fine rows,
// plus kMargin, as half-width.
__global__ void k_width_target(const int32_t* __restrict__ cpath, const int* __restrict__ clen,
                               const int32_t* __restrict__ path, const int* __restrict__ plen,
                               int ds, int Lac, float wmin, float wmax, float* __restrict__ wt) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= Lac) return;
    const int nc = *clen, nf = *plen;
    float need = 0.f;
    if (nc > 0) {
        const int lo = first_of_row(cpath, nc, i - 1);
        int jmin = 0x7fffffff, jmax = -1;
        for (int k = lo; k < nc && cpath[2 * k] <= i + 1; ++k) {
            jmin = min(jmin, cpath[2 * k + 1]);
            jmax = max(jmax, cpath[2 * k + 1]);
        }
        const int f0 = jmin * ds, f1 = (jmax + 1) * ds - 1;
        for (int k = first_of_row(path, nf, i * ds); k < nf && path[2 * k] < (i + 1) * ds; ++k) {
            const int j = path[2 * k + 1];
            need = fmaxf(need, (float)max(max(f0 - j, j - f1), 0));
        }
    } else {
        need = wmax;
    }
    const float t = log2f((need + kMargin) / wmin) / log2f(wmax / wmin);
    wt[i] = fminf(fmaxf(t, 0.f), 1.f);
}

// Pinball loss of sigmoid(s_i) against wt_i at quantile kQ (mean over rows);
// ds[i] = dL/ds_i.
__global__ void k_loss_width(const float* __restrict__ S, const float* __restrict__ wt, int Lac,
                             float* __restrict__ dS, float* __restrict__ loss) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= Lac) return;
    const float p = 1.f / (1.f + expf(-S[i]));
    const float d = wt[i] - p;
    const float inv_n = 1.f / (float)Lac;
    atomicAdd(loss, (d > 0.f ? kQ * d : (kQ - 1.f) * d) * inv_n);
    const float dp = d > 0.f ? -kQ : (1.f - kQ);
    dS[i] = dp * p * (1.f - p) * inv_n;
}

// Adam (bias-corrected), then the gradient is zeroed for the next step.
__global__ void k_adam(int n, float* __restrict__ P, float* __restrict__ G, float* __restrict__ M,
                       float* __restrict__ V, float lr, float b1, float b2, float eps, float c1,
                       float c2) {
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= n) return;
    const float g = G[k];
    const float m = b1 * M[k] + (1.f - b1) * g;
    const float v = b2 * V[k] + (1.f - b2) * g * g;
    M[k] = m;
    V[k] = v;
    P[k] -= lr * (m / c1) / (sqrtf(v / c2) + eps);
    G[k] = 0.f;
}

// Grid of both sequences of q in tiles of `rows` rows.
template <class Q>
dim3 enc_grid(const Q& q, int n, int rows, int y = 1) {
    int L = 0;
    for (int k = 0; k < n; ++k) L = q.s[k].L > L ? q.s[k].L : L;
    return dim3((unsigned)((L + rows - 1) / rows), (unsigned)y, (unsigned)n);
}

template <bool kBwd, bool kBF16>
cudaError_t conv_t(const EncRows2& q, int n, int Cin, const float* W, const float* b, int relu,
                   cudaStream_t s) {
    static_assert((kC * kXS + kC * kK * kWS) * 4 <= 48 * 1024, "default shared memory");
    const int smem = (Cin * kXS + Cin * kK * kWS) * (int)sizeof(float);
    const dim3 grid = enc_grid(q, n, kTL, kC / kCO);
    if (Cin == kC)
        k_conv<kC, kBwd, kBF16><<<grid, kConvThreads, smem, s>>>(q, Cin, W, b, relu);
    else
        k_conv<0, kBwd, kBF16><<<grid, kConvThreads, smem, s>>>(q, Cin, W, b, relu);
    return cudaGetLastError();
}

}  // namespace

EncLayout enc_layout(int D) {
    EncLayout p;
    size_t o = 0;
    p.W1 = o; o += (size_t)kC * D * kK;
    p.b1 = o; o += kC;
    p.W2 = o; o += (size_t)kC * kC * kK;
    p.b2 = o; o += kC;
    p.W3 = o; o += (size_t)kC * kC * kK;
    p.b3 = o; o += kC;
    p.W4 = o; o += (size_t)kE * kC;
    p.b4 = o; o += kE;
    p.W5 = o; o += kC;
    p.b5 = o; o += 1;
    p.count = o;
    return p;
}

cudaError_t launch_pool_norm(const EncRows2& q, int n, int D, int ds, cudaStream_t s) {
    if (D < 1 || D > kC) return cudaErrorInvalidValue;
    EncRows2 c = q;  // coarse rows for the grid
    for (int k = 0; k < n; ++k) c.s[k].L = (q.s[k].L + ds - 1) / ds;
    if (D <= 16)
        k_pool_norm<16><<<enc_grid(c, n, 8), 128, 0, s>>>(q, D, ds);
    else
        k_pool_norm<32><<<enc_grid(c, n, 4), 128, 0, s>>>(q, D, ds);
    return cudaGetLastError();
}

cudaError_t launch_conv(const EncRows2& q, int n, int Cin, const float* W, const float* b, int relu,
                        int bwd, int bf16, cudaStream_t s) {
    if (Cin < 1 || Cin > kC) return cudaErrorInvalidValue;
    if (bwd) return bf16 ? cudaErrorInvalidValue : conv_t<true, false>(q, n, Cin, W, b, relu, s);
    return bf16 ? conv_t<false, true>(q, n, Cin, W, b, relu, s)
                : conv_t<false, false>(q, n, Cin, W, b, relu, s);
}

cudaError_t launch_conv_wgrad(const EncGrad2& q, int n, int Cin, float* dW, float* db,
                              cudaStream_t s) {
    if (Cin < 1 || Cin > kC) return cudaErrorInvalidValue;
    k_conv_wgrad<<<enc_grid(q, n, kTW * kTiles, (Cin + kCI - 1) / kCI), kWgThreads, 0, s>>>(q, Cin, dW, db);
    return cudaGetLastError();
}

cudaError_t launch_embed(const EncEmbed2& q, int n, const float* params, const EncLayout& p, int bf16,
                         float wmin, float wmax, cudaStream_t s) {
    k_embed<<<enc_grid(q, n, 32), 128, 0, s>>>(q, params + p.W4, params + p.b4, params + p.W5,
                                              params + p.b5, bf16, wmin, wmax);
    return cudaGetLastError();
}

cudaError_t launch_embed_bwd(const EncEmbed2& q, int n, const float* W4, cudaStream_t s) {
    k_embed_bwd<<<enc_grid(q, n, kBwdRows), 256, 0, s>>>(q, W4);
    return cudaGetLastError();
}

cudaError_t launch_head_grad(const EncHead2& q, int n, int outputs, float* dW, float* db,
                             cudaStream_t s) {
    if (outputs == kE)
        k_head_grad<kE><<<enc_grid(q, n, kHeadRows), 256, 0, s>>>(q, dW, db);
    else if (outputs == 1)
        k_head_grad<1><<<enc_grid(q, n, kHeadRows), 256, 0, s>>>(q, dW, db);
    else
        return cudaErrorInvalidValue;
    return cudaGetLastError();
}

cudaError_t launch_targets(const int32_t* path, const int* plen, int cap, int ds, int Lac,
                           unsigned long long* jsum, int* cnt, cudaStream_t s) {
    k_targets<<<(cap + 127) / 128, 128, 0, s>>>(path, plen, cap, ds, Lac, jsum, cnt);
    return cudaGetLastError();
}

cudaError_t launch_loss_emb(const float* eA, int Lac, const float* eB, int Lbc,
                            const unsigned long long* jsum, const int* cnt, int ds, float* gA,
                            float* gB, float* loss, cudaStream_t s) {
    k_loss_emb<<<(Lac + kLossRows - 1) / kLossRows, 32 * kLossRows, 0, s>>>(
        eA, Lac, eB, Lbc, jsum, cnt, ds, gA, gB, loss);
    return cudaGetLastError();
}

cudaError_t launch_width_target(const int32_t* cpath, const int* clen, const int32_t* path,
                                const int* plen, int ds, int Lac, float wmin, float wmax,
                                float* wt, cudaStream_t s) {
    k_width_target<<<(Lac + 127) / 128, 128, 0, s>>>(cpath, clen, path, plen, ds, Lac, wmin, wmax,
                                                     wt);
    return cudaGetLastError();
}

cudaError_t launch_loss_width(const float* S, const float* wt, int Lac, float* dS, float* loss,
                              cudaStream_t s) {
    k_loss_width<<<(Lac + 255) / 256, 256, 0, s>>>(S, wt, Lac, dS, loss);
    return cudaGetLastError();
}

cudaError_t launch_adam(int n, float* P, float* G, float* M, float* V, int step, float lr,
                        float b1, float b2, float eps, cudaStream_t s) {
    const float c1 = 1.f - powf(b1, (float)step), c2 = 1.f - powf(b2, (float)step);
    k_adam<<<(n + 255) / 256, 256, 0, s>>>(n, P, G, M, V, lr, b1, b2, eps, c1, c2);
    return cudaGetLastError();
}

}  // namespace pardtw

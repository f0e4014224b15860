// Internal declarations shared by the CUDA translation units of libpardtw.
// Not part of the public C-ABI (include/pardtw.h).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <atomic>

#include "pardtw.h"

namespace pardtw {

// Launch facts of a kernel that are per device: its dynamic shared memory
// limit (cudaFuncSetAttribute applies to the current device) and the CTAs of
// it resident per SM.  Each launcher keeps one DeviceSlots per kernel
// instantiation (static storage: zero-initialised, 0 = not looked up yet).
constexpr int kMaxDevices = 64;
struct DeviceSlots {
    std::atomic<int> v[kMaxDevices];
};

// Raise `kern`'s dynamic shared memory limit to `smem` bytes on the current
// device, once per device.
template <class K>
cudaError_t raise_smem_once(K* kern, int smem, DeviceSlots& done) {
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    const bool slot = dev >= 0 && dev < kMaxDevices;
    if (slot && done.v[dev].load(std::memory_order_acquire) != 0) return cudaSuccess;
    e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e != cudaSuccess) return e;
    if (slot) done.v[dev].store(1, std::memory_order_release);
    return cudaSuccess;
}

// CTAs of `kern` (threads a CTA, smem bytes of dynamic shared memory)
// resident per SM of the current device, at least 1; raises the kernel's
// shared memory limit there first.  Looked up once per device.
template <class K>
cudaError_t blocks_per_sm_once(K* kern, int threads, int smem, DeviceSlots& cache, int* out) {
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    const bool slot = dev >= 0 && dev < kMaxDevices;
    if (slot) {
        const int n = cache.v[dev].load(std::memory_order_acquire);
        if (n > 0) {
            *out = n;
            return cudaSuccess;
        }
    }
    e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e != cudaSuccess) return e;
    int n = 0;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, kern, threads, smem);
    if (e != cudaSuccess) return e;
    if (n < 1) n = 1;
    if (slot) cache.v[dev].store(n, std::memory_order_release);
    *out = n;
    return cudaSuccess;
}

// Kernels of one call in a chain: each is launched with launch_chained, so that
// its CTAs are placed while the kernel before it in the stream still runs, and
// starts with chain_wait (all its threads, before the first access to global
// memory), which returns when that kernel has completed and its writes can be
// seen; chain_next then lets the kernel behind it be placed.  As it comes after
// the wait, a kernel that runs has only its direct predecessor in flight beside
// it: what older kernels of the chain wrote may be read through the read-only
// path, the direct predecessor's results may not (a plain load).  The first kernel
// of a call is launched plainly, behind everything in its stream, and only
// calls chain_next.
__device__ __forceinline__ void chain_wait() {
    asm volatile("griddepcontrol.wait;" ::: "memory");
}
__device__ __forceinline__ void chain_next() {
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}
inline cudaLaunchAttribute chained_attr(bool chained) {
    cudaLaunchAttribute at = {};
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = chained ? 1 : 0;
    return at;
}
// (chained false: an ordinary launch)
template <class... P, class... A>
cudaError_t launch_chained(bool chained, void (*kern)(P...), dim3 grid, int threads, int smem,
                           cudaStream_t s, const A&... args) {
    cudaLaunchAttribute at = chained_attr(chained);
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = dim3((unsigned)threads);
    cfg.dynamicSmemBytes = (size_t)smem;
    cfg.stream = s;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    const cudaError_t e = cudaLaunchKernelEx(&cfg, kern, static_cast<P>(args)...);
    if (e != cudaSuccess) (void)cudaGetLastError();
    return e;
}

constexpr int kWarp = 32;
constexpr long long kDefaultTimeoutNs = 2000000000LL;  // bounded device waits: 2 s
constexpr int kRowsPerStrip = 30;   // rows of A per warp: lanes 0..29 (lanes 30, 31 carry
                                    // the two bottom rows of the strip above)
constexpr int kColsPerWord = 16;    // 2-bit codes per uint32 backpointer word
constexpr int kWarpsPerGroup = 4;   // strips per CTA ("strip group") of the one-warp kernels
constexpr int kSplitStrips = 2;     // strips per CTA of the cost/DP warp-pair kernel
// CTAs of the warp-pair DP kernel (without clusters) to be resident per SM: two
// where the registers allow it (two strips per CTA, up to 3 rows per lane and
// R x dp <= 36), which the kernel's launch bounds then enforce, else one.
__host__ __device__ constexpr int split_ctas_per_sm(int R, int ns, int dp, bool bf16) {
    return (ns == 2 && !bf16 && R <= 3 && R * dp <= 36) ? 2 : 1;
}
// BF16 cost (tensor cores): a frame of B (or row of A) takes kBfStride bf16
// in memory, 128 features and 8 of padding, so that the 8 rows an ldmatrix
// reads start 272 bytes apart, in 8 different bank groups.
constexpr int kBfStride = 136;

// Device status words (workspace).  [0] first error (DTW_* code), [1] detail,
// [2] ticket counter of the persistent DP kernel, [3] spare.
struct DevCtl {
    int status;
    int detail;
    int ticket;
    int spare;
};

// Arguments of the column-sweep DP kernel.
struct DpArgs {
    const float* Ahat;              // nstrips*30 x dp, row-normalised, rows >= La are zero
    const float* Bhat;              // row-normalised B, chunk-transposed (see bt_index)
    const void* Bbf;                // BF16 cost only: normalised B as bf16, frame-major,
                                    // kBfStride elements per frame (else null)
    uint32_t* bp;                   // nstrips * nchunk * 32 words (strip, chunk, row in strip)
    unsigned long long* gborder;    // ngroups * Lb * 2 tagged values (group bottom rows)
    DevCtl* ctl;
    float* e_final;                 // shifted cumulative cost at (La-1, Lb-1)
    int La, Lb;
    int nstrips, nchunk, ngroups;
    int rps;                        // rows of A per strip (warp)
    int wpb;                        // backpointer words per (strip, 16 columns)
    float kcost;                    // 1 - cost_shift
    float mu;                       // cost_shift
    unsigned epoch;                 // call tag for global border entries
    long long timeout_ns;
    int skip_publish;               // group that never publishes (fault injection), -1 off
    int feats;                      // features of a frame; those up to the padded width are zero
    const int2* ranges;             // banded DP (warp-pair kernel): per strip the sub-chunks
                                    // [x, y) of 8 columns it sweeps (x even; x and y
                                    // non-decreasing in the strip); null = the columns
                                    // that a path can cross (subsequence DP: every column)
    float* lastrow;                 // subsequence DP (WSDTW): the cumulative cost of row
                                    // La-1 at every column (nchunk * 16 floats), else null
};

// Columns of row i that a path can cross, [path_lo, path_hi]: with steps of
// slope 1/2 to 2, the cells reachable from (0, 0) that can still reach
// (La-1, Lb-1).  Both bounds grow with i, and every predecessor a path can
// take lies inside them, so cells outside (two thirds of a square matrix)
// never change a path, a total or a field that a path reads.
__host__ __device__ inline int path_lo(int i, int La, int Lb) {
    const int a = (i + 1) / 2, b = Lb - 1 - 2 * (La - 1 - i);
    return a > b ? a : b;
}
__host__ __device__ inline int path_hi(int i, int La, int Lb) {
    const int a = 2 * i, b = Lb - 1 - (La - i) / 2;
    return a < b ? a : b;
}

// Backpointer word address of cell (i, j): strip-major, then 16-column chunk,
// then row within the strip.  A strip of rps rows stores wpb >= rps words
// per chunk (32 per warp and row of a lane: the ghost lane's words are
// unused), so one warp store covers wpb consecutive words.
__host__ __device__ inline size_t bp_word_index(int i, int j, int nchunk, int rps, int wpb) {
    const int strip = i / rps;
    return ((size_t)strip * (size_t)nchunk + (size_t)(j >> 4)) * (size_t)wpb +
           (size_t)(i - strip * rps);
}

// Backpointer field of cell (i, j): 2 bits at bit 2 * (j % 16) of its word.
// Bit 0 is set when the (1,1) candidate attains the cell's minimum, bit 1
// when the (1,2) candidate does.  The step taken is the first attaining
// candidate in the order (1,1), (1,2), (2,1) (a later candidate must be
// strictly smaller), so: bit 0 set -> (1,1); field 2 -> (1,2); field 0 ->
// (2,1).  Returns the step code 0 = (1,1), 1 = (1,2), 2 = (2,1).
__host__ __device__ inline int step_of_field(uint32_t field) {
    return (field & 1u) ? 0 : (field == 2u ? 1 : 2);
}

// Strip geometry of the DP kernels: R rows per lane.  R = 1: lanes 0..29
// are rows, lanes 30, 31 carry the strip above (30 rows, 32 words).  R >= 2:
// lanes 0..30 hold R rows each, lane 31 carries the strip above (31 R rows,
// 32 R words).
__host__ __device__ inline int strip_rows(int R) { return R == 1 ? 30 : 31 * R; }
__host__ __device__ inline int strip_words(int R) { return 32 * R; }

// Normalised frames of B are stored chunk-transposed: 16 consecutive frames
// (one backpointer chunk) form a feature-major block of 16 * dp floats, so
// value d of frame f sits at ((f / 16) * dp + d) * 16 + f % 16.  A partial
// last chunk is zero-padded.  The DP kernel reads these blocks feature by
// feature to spread the 16 cost computations of a chunk over its steps.
__host__ __device__ inline size_t bt_index(int f, int d, int dp) {
    return ((size_t)(f >> 4) * (size_t)dp + (size_t)d) * 16u + (size_t)(f & 15);
}

// Normalisation of one pair.
struct NormArgs {
    const float* A;
    int La, La_pad;
    const float* B;
    int Lb, Lb_pad;
    float* Ahat;
    float* Bt;
    DevCtl* ctl;
};

// Launchers (each returns a cudaError_t from the launch).
// Bbf: null, or for the BF16 cost B normalised as bf16 instead of Bt: Lb_pad
// frames of kBfStride elements (features beyond D and frames beyond Lb are zero).
cudaError_t launch_normalise(const NormArgs& a, int D, int dp, void* Bbf, cudaStream_t s);
cudaError_t launch_cost(const float* Ahat, int La, const float* Bt, int Lb, int dp, float* C,
                        cudaStream_t s);
// n pairs at once (`many`: device array); max_blocks = the most
// normalise_blocks(La_pad, Lb_pad) among them; also zeroes *ticket, the work
// queue of launch_dp_split_many.
cudaError_t launch_normalise_many(const NormArgs* many, int n, int max_blocks, int D, int dp,
                                  int* ticket, cudaStream_t s);
int normalise_blocks(int La_pad, int Lb_pad);
// Every DpArgs::epoch of a batch in device memory += 1 (0 skipped).
cudaError_t launch_bump_epoch(DpArgs* many, int n, cudaStream_t s);
cudaError_t launch_dp(const DpArgs& a, int dp, int num_sms, cudaStream_t s);           // R = 1
cudaError_t launch_dp_multirow(const DpArgs& a, int dp, int R, int num_sms, cudaStream_t s);
// Rows per lane the fused DP supports for a padded dimension (0 = none).
bool multirow_supported(int dp, int R);
// Warp-specialised DP (dp_split.cu, dp_split4.cu): a cost warp and a DP warp
// per strip, ns = 2 or 4 strips per CTA; R = 2, 3 or 4 rows per lane.
// transposed: the pair is swept with A and B swapped (rows of the kernel =
// frames of B), with the tie order mapped back (R = 3, one pair).
cudaError_t launch_dp_split(const DpArgs& a, int dp, int R, int ns, int num_sms, cudaStream_t s,
                            bool transposed = false);
bool split4_supported(int dp, int R);
cudaError_t launch_dp_split4(const DpArgs& a, const DpArgs* many, const int2* queue, int items,
                             int* ticket, int dp, int R, int num_sms, cudaStream_t s,
                             bool transposed);
// The subsequence DP of WSDTW over a batch (R = 3, dp <= 32): weights 1, 1, 2,
// free start in row 0, row La-1 of every pair into its DpArgs::lastrow.
cudaError_t launch_dp_subseq_many(const DpArgs* many, const int2* queue, int items,
                                  int* ticket, int dp, int num_sms, cudaStream_t s);
// ns strips per CTA: 2 (every dp <= 32) or 4 (dp <= 16, R = 2, 3).
bool split_supported(int dp, int R, int ns = 2);
// The same DP with the cost from BF16 features and FP32 accumulation on the
// tensor cores (mma.sync m16n8k16): D padded to 64 or 128, R = 3.
cudaError_t launch_dp_split_bf16(const DpArgs& a, int dp, int num_sms, cudaStream_t s,
                                 bool transposed = false);
// The warp-pair DP of one pair at 3 rows per lane, run in thread-block clusters whose
// CTAs pass the strip border through distributed shared memory (dp_split_cl.cu; two
// strips per CTA at dp <= 16, one at 32 and, FP32 or bf16, at 64 and 128).
// *used = false (and nothing launched) when no cluster configuration fits
// this device.
cudaError_t launch_dp_split_cl(const DpArgs& a, int dp, bool bf16, bool transposed,
                               cudaStream_t s, bool* used);
// The warp-pair DP with the FP32 cost at D = 64, 128 (dp_split_wide.cu), 3 rows per
// lane: two strips per CTA with two cost warps each; in thread-block clusters one
// with four.
bool split_wide_supported(int dp);
cudaError_t launch_dp_split_wide(const DpArgs& a, int dp, int num_sms, cudaStream_t s,
                                 bool transposed = false);
cudaError_t launch_dp_split_wide_cl(const DpArgs& a, int dp, bool transposed, cudaStream_t s,
                                    bool* used);
bool split_bf16_supported(int dp);
// Many pairs in one persistent launch: `many` (device) holds the pairs' DpArgs,
// queue (device) the `items` (pair, strip group) items in the order CTAs take
// them from *ticket; a pair's groups stand in ascending order, so a group only
// waits on groups of its own pair that were taken earlier.  Each pair's
// failures stay in its own control block.
cudaError_t launch_dp_split_many(const DpArgs* many, const int2* queue, int items, int* ticket,
                                 int dp, int R, int ns, int num_sms, cudaStream_t s);

// Which DP kernel runs a problem: kind 0 = one row per lane (dp_kernel.cu),
// 1 = fused multi-row (dp_multirow.cu), 2 = cost/DP warp pairs (dp_split.cu);
// R rows per lane, spg strips per CTA (strip group).
struct DpPlan {
    int kind, R, spg;
    int bf16;  // kind 2 only: the cost on the tensor cores from BF16 features
    int no_clusters;  // kind 2, R = 3, two strips: 1 = never run in thread-block clusters
};
DpPlan choose_plan(int La, int dp, const dtw_options& o, int num_sms);
// Whether a pair is swept transposed (B's frames as rows): B longer than A
// (or forced by the options) and the transposed pair's plan is the warp-pair
// DP at 3 rows per lane.
bool transpose_pair(int La, int Lb, int dp, const dtw_options& o, int num_sms);
cudaError_t launch_plan(const DpPlan& plan, const DpArgs& a, int dp, int num_sms,
                        cudaStream_t s, bool transposed = false);

// Bytes to allocate for a handle's buffer that needs `need` and had `had`: room for an
// eighth more, so that a handle fed growing pairs synchronises and allocates anew once per
// eighth; none in a first small allocation, which then shares its mapping with
// others (first call of 1000 x 1200 frames: 217 us with a mapping of its own, 119).
size_t grown_bytes(size_t need, size_t had);

// Parallel backtrace through per-band entry maps (bandmap.cu) of one pair:
// its backpointers and layout, its control block and end cell, the outputs,
// and caller-provided scratch of bandmap_scratch_bytes(La, Lb) bytes.
struct BtArgs {
    const uint32_t* bp;
    int La, Lb, nchunk, rps, wpb;
    DevCtl* ctl;
    const float* e_final;
    float mu;
    int32_t* path;
    int* path_len;
    float* total;
    void* scratch;
    const int2* ranges;  // banded DP: the strips' sub-chunk ranges (cells outside have no
                         // path), else null
    int transposed;      // the matrix is the transposed problem's: emit (column, row)
    int band;            // rows per band: band_rows(La, cells)
    int chained;         // set by launch_backtrace_bands: its kernels form a chain
};
// Rows per band of a pair of La rows in a call over `cells` matrix cells in all:
// the band map and the walks take time in proportion to a band's rows (~0.17 and
// ~0.06 us a row, all bands at once), the chain in proportion to the number of
// bands (~0.6 us for four), so short pairs take short bands (1000 x 1200: 96.9 us
// with 128 rows, 82.6 with 32; 3001 x 3607: 216 and 206 with 64) unless the call
// fills the GPU: a segment of the map recomputes two columns per row of its band (256
// pairs of up to 8000 frames: 3.66 ms with 64 rows, 3.51 with 128).
inline int band_rows(int La, double cells) {
    if (cells > 1e9) return 128;
    return La <= 1536 ? 32 : (La <= 6144 ? 64 : 128);
}
size_t bandmap_scratch_bytes(int La, int Lb);
cudaError_t launch_backtrace_bands(const BtArgs& a, cudaStream_t s);
// n pairs at once; `many` is a device array of n BtArgs, nbands and maxLb the
// most bands and columns among them.
cudaError_t launch_backtrace_bands_many(const BtArgs* many, int n, int nbands, int maxLb,
                                        cudaStream_t s);

// Padded feature width used by the kernels for a given D (0 = unsupported).
int padded_dim(int D);

// Multiscale band (band.cu): Y (ceil(L/ds) x D) = averages of ds frames of X;
// per strip of rps fine rows the 8-column blocks within w columns of the
// coarse path (cpath, *clen cells) scaled by ds, widened to monotone; *touch
// = 1 if the banded path (path, *plen cells) comes within one block of a
// side of the band that is not the side of the matrix.
// wrow (may be null): per coarse row of A a half-width in fine frames that
// replaces w (the largest over the coarse rows next to a strip is used).
cudaError_t launch_pool(const float* X, int L, int D, int ds, float* Y, cudaStream_t s);
// swap: the fine DP sweeps the transposed pair (paths are read as (j, i);
// La, Lb, Lac are the swept pair's rows, columns, coarse rows).
cudaError_t launch_band_ranges(const int32_t* cpath, const int* clen, int ds, int w,
                               const float* wrow, int Lac, int La, int Lb, int nstrips, int rps,
                               int swap, int2* ranges, cudaStream_t s);
cudaError_t launch_band_touch(const int32_t* path, const int* plen, int cap, int Lb, int rps,
                              const int2* ranges, int swap, int* touch, cudaStream_t s);

// WSDTW (wsdtw.cu): one fragment of A, its backtrace matrix from the batched
// subsequence DP and the control block of its DP.
struct WsFrag {
    const uint32_t* bp;
    const DevCtl* pctl;
    int row0, len;          // first row of A, rows
    int nchunk, rps, wpb;   // backtrace matrix geometry (see bp_word_index)
};
// Segment-level DP over the fragments' last rows (stride floats apart) with
// shortest matches delta[k]; end frames, total (D_seg[N-1][Lb-1]) and status.
// agg: seg_dp_scratch_bytes(Lb) bytes; done: two counters (zeroed here);
// timeout_ns bounds each wait of the one-grid form.
cudaError_t launch_seg_dp(const WsFrag* fr, const float* lastrow, size_t stride, int N, int Lb,
                          const int* delta, float* Dseg, int* arg, void* agg, unsigned* done,
                          int* ends, float* total, DevCtl* ctl, long long timeout_ns,
                          cudaStream_t s);
size_t seg_dp_scratch_bytes(int Lb);
// Fragment backtraces from their end frames into `scratch` (2 La ints), then
// the concatenated path into `path` and its length (or -status) into path_len.
cudaError_t launch_bt_subseq(const WsFrag* fr, int N, const int* ends, int32_t* scratch,
                             int* count, int32_t* path, int* path_len, DevCtl* ctl,
                             cudaStream_t s);

// Band encoder (encoder.cu).  Parameter offsets (floats) of the flat
// parameter array for input dimension D; see pardtw.h for the layout.
constexpr int kEncChannels = 64;
constexpr int kEncEmbed = 16;
constexpr int kEncKernel = 5;
struct EncLayout {
    size_t W1, b1, W2, b2, W3, b3, W4, b4, W5, b5, count;
};
EncLayout enc_layout(int D);
// A layer's rows of one or two sequences (n of them; one launch runs both).
struct EncRows {
    const float* X;  // input rows
    const float* M;  // conv backward: rows of X count where M > 0 (may be null)
    float* Y;        // output rows
    int L;
};
struct EncGrad {
    const float *X, *dY, *Yout;
    int L;
};
struct EncEmbed {
    const float* H;
    float *Emb, *invn, *S, *HW, *G, *dH;  // see k_embed, k_embed_bwd
    int L;
    unsigned long long* jsum;  // see k_targets
    int* cnt;
};
struct EncHead {
    const float *U, *H;
    int L;
};
struct EncRows2 { EncRows s[2]; };
struct EncGrad2 { EncGrad s[2]; };
struct EncEmbed2 { EncEmbed s[2]; };
struct EncHead2 { EncHead s[2]; };
// X: fine frames (L of them), Y: pooled, normalised frames.
cudaError_t launch_pool_norm(const EncRows2& q, int n, int D, int ds, cudaStream_t s);
// conv5 of L rows: forward (bwd = 0: W [64][Cin][5], bias, relu) or the
// backward-data pass (bwd = 1: W the forward weight [64][64][5] read
// transposed and flipped, X masked by M > 0); bf16 rounds inputs and
// weights (forward only).
cudaError_t launch_conv(const EncRows2& q, int n, int Cin, const float* W, const float* b, int relu,
                        int bwd, int bf16, cudaStream_t s);
cudaError_t launch_conv_wgrad(const EncGrad2& q, int n, int Cin, float* dW, float* db,
                              cudaStream_t s);
cudaError_t launch_embed(const EncEmbed2& q, int n, const float* params, const EncLayout& p, int bf16,
                         float wmin, float wmax, cudaStream_t s);
cudaError_t launch_embed_bwd(const EncEmbed2& q, int n, const float* W4, cudaStream_t s);
// outputs = 16 (embedding head) or 1 (half-width head).
cudaError_t launch_head_grad(const EncHead2& q, int n, int outputs, float* dW, float* db,
                             cudaStream_t s);
// jsum, cnt: Lac each, added to (zeroed by launch_embed).
cudaError_t launch_targets(const int32_t* path, const int* plen, int cap, int ds, int Lac,
                           unsigned long long* jsum, int* cnt, cudaStream_t s);
// gB is added to (zeroed by launch_embed's G).
cudaError_t launch_loss_emb(const float* eA, int Lac, const float* eB, int Lbc,
                            const unsigned long long* jsum, const int* cnt, int ds, float* gA,
                            float* gB, float* loss, cudaStream_t s);
cudaError_t launch_width_target(const int32_t* cpath, const int* clen, const int32_t* path,
                                const int* plen, int ds, int Lac, float wmin, float wmax,
                                float* wt, cudaStream_t s);
cudaError_t launch_loss_width(const float* S, const float* wt, int Lac, float* dS, float* loss,
                              cudaStream_t s);
cudaError_t launch_adam(int n, float* P, float* G, float* M, float* V, int step, float lr,
                        float b1, float b2, float eps, cudaStream_t s);

}  // namespace pardtw

// Weakly-ordered Segmental DTW (WSDTW, Sec. II-C), steps 3 to 5 on the GPU.
// Steps 1 and 2 (the fragments of A and their subsequence DTW against all of
// B) run in the batched warp-pair DP (dp_split.cu, subsequence mode), which
// leaves every fragment's last row of cumulative costs (C_seg, step 3) and its
// 2-bit backtrace matrix.  Here:
//
//   k_seg_tile,  step 4, fragment k = 0 .. N-1 in turn (two launches each):
//   k_seg_fix      match[j]   = D_seg[k-1][j - delta_k] + C_seg[k][j]
//                               (= C_seg[0][j] for k = 0; +inf for j < delta_k)
//                  D_seg[k][j] = running minimum of match over j' <= j,
//                  arg[k][j]   = the first j' attaining it,
//                as a tiled prefix scan; then the end frames
//                e_{N-1} = arg[N-1][Lb-1], e_{k-1} = arg[k-1][e_k - delta_k].
//   k_seg_cluster, k_seg_all   the same in one launch: in one cluster, or in one grid
//   k_bt_subseq  step 5, one warp per fragment: the walk from (last row,
//                e_k) back to row 0 through the fragment's backtrace matrix,
//                written backwards into the fragment's slots of a scratch path.
//   k_compact    the fragment paths one after another into the caller's path.
#include <atomic>

#include "dp_device.cuh"
#include "block_walk.cuh"

namespace pardtw {

namespace {

constexpr int kCompactThreads = 256;

// (value, index) minimum where the earlier index wins ties.
struct MinArg {
    float v;
    int j;
};
__device__ __forceinline__ MinArg better(MinArg a, MinArg b) {  // a is earlier
    return (b.v < a.v) ? b : a;
}

// Step 4 runs fragment by fragment; within fragment k the running minimum
// over j is a prefix scan of (value, column) pairs (the earlier column wins
// ties), done in tiles of kTile columns by two launches:
//   k_seg_tile   every tile: its match values (coalesced), their minimum into
//                agg[tile]; the last tile to finish (a counter, no waiting)
//                turns agg into exclusive carries for all tiles;
//   k_seg_fix    every tile: the block-wide inclusive scan of its match values
//                from its carry, written as D_seg[k][*] and arg[k][*].
constexpr int kTile = 1024;

// A match that is NaN (a frame that is) is never attained: +inf, in every form of this DP.
__device__ __forceinline__ float attainable(float match) { return fminf(match, INFINITY); }

__device__ __forceinline__ float seg_match(const float* cs, const float* prev, int k, int dk,
                                           int j) {
    if (k == 0) return attainable(cs[j]);
    return j - dk >= 0 ? attainable(prev[j - dk] + cs[j]) : INFINITY;
}

// Block-wide inclusive scan of one (value, column) per thread, earlier wins.
__device__ __forceinline__ MinArg block_scan_min(MinArg v, MinArg* s_warp) {
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
        MinArg o;
        o.v = __shfl_up_sync(0xffffffffu, v.v, off);
        o.j = __shfl_up_sync(0xffffffffu, v.j, off);
        if (lane >= off) v = better(o, v);
    }
    if (lane == 31) s_warp[w] = v;
    __syncthreads();
    if (w == 0) {
        MinArg x = lane < (int)(blockDim.x >> 5) ? s_warp[lane] : MinArg{INFINITY, -1};
#pragma unroll
        for (int off = 1; off < 32; off <<= 1) {
            MinArg o;
            o.v = __shfl_up_sync(0xffffffffu, x.v, off);
            o.j = __shfl_up_sync(0xffffffffu, x.j, off);
            if (lane >= off) x = better(o, x);
        }
        s_warp[lane] = x;  // inclusive prefix over warps
    }
    __syncthreads();
    if (w > 0) v = better(s_warp[w - 1], v);
    return v;
}

__global__ void __launch_bounds__(kTile)
    k_seg_tile(const WsFrag* __restrict__ fr, const float* __restrict__ lastrow, size_t stride,
               int N, int Lb, int k, const int* __restrict__ delta,
               const float* __restrict__ Dseg, MinArg* __restrict__ agg,
               unsigned* __restrict__ done, DevCtl* ctl) {
    __shared__ MinArg s_warp[32];
    __shared__ bool s_last;
    const int ntile = gridDim.x;
    const int j = blockIdx.x * kTile + threadIdx.x;
    const float* cs = lastrow + (size_t)k * stride;
    const float* prev = k > 0 ? Dseg + (size_t)(k - 1) * Lb : nullptr;
    const int dk = k > 0 ? delta[k] : 0;
    MinArg v{INFINITY, -1};
    if (j < Lb) v = MinArg{seg_match(cs, prev, k, dk, j), j};
    v = block_scan_min(v, s_warp);
    if (threadIdx.x == blockDim.x - 1) {
        agg[blockIdx.x] = v;
        __threadfence();
        s_last = atomicAdd(done, 1u) == (unsigned)ntile - 1;
    }
    __syncthreads();
    if (!s_last) return;
    // the last tile: exclusive carries of all tiles, in tile order (a few
    // hundred tiles at most), then the counter is reset for the next launch
    __threadfence();
    if (threadIdx.x == 0) {
        // a fragment whose DP failed (a bounded wait expired) fails the call
        if (k == 0)
            for (int q = 0; q < N; ++q) {
                const int st = fr[q].pctl->status;
                if (st != 0) {
                    raise_status(ctl, st, 20);
                    break;
                }
            }
        MinArg run{INFINITY, -1};
        volatile MinArg* va = agg;  // written by the other tiles of this launch
        for (int t = 0; t < ntile; ++t) {
            const MinArg a{va[t].v, va[t].j};
            va[t].v = run.v;  // carry into tile t
            va[t].j = run.j;
            run = better(run, a);
        }
        *done = 0u;
    }
}

__global__ void __launch_bounds__(kTile)
    k_seg_fix(const float* __restrict__ lastrow, size_t stride, int N, int Lb, int k,
              const int* __restrict__ delta, float* __restrict__ Dseg, int* __restrict__ arg,
              const MinArg* __restrict__ agg, int* __restrict__ ends, float* __restrict__ total,
              DevCtl* ctl) {
    __shared__ MinArg s_warp[32];
    const int j = blockIdx.x * kTile + threadIdx.x;
    const float* cs = lastrow + (size_t)k * stride;
    const float* prev = k > 0 ? Dseg + (size_t)(k - 1) * Lb : nullptr;
    const int dk = k > 0 ? delta[k] : 0;
    MinArg v{INFINITY, -1};
    if (j < Lb) v = MinArg{seg_match(cs, prev, k, dk, j), j};
    v = better(agg[blockIdx.x], block_scan_min(v, s_warp));
    if (j < Lb) {
        Dseg[(size_t)k * Lb + j] = v.v;
        arg[(size_t)k * Lb + j] = v.j;
    }
    // the last fragment's last column: the total and the end frames
    if (k == N - 1 && j == Lb - 1) {
        if (ctl->status != 0) return;
        if (!(v.v < INFINITY)) {
            raise_status(ctl, DTW_ERR_UNREACHABLE, 21);
            return;
        }
        *total = v.v;
        int e = v.j;
        ends[N - 1] = e;
        for (int q = N - 1; q > 0; --q) {
            e = arg[(size_t)(q - 1) * Lb + (e - delta[q])];
            ends[q - 1] = e;
        }
    }
}

// One warp per fragment: the subsequence path from (len-1, e_k) to row 0
// (WindowWalker), stored backwards (ascending once read from slot
// row0 + len - n) as global (row of A, frame of B) pairs.  A step that
// leaves the fragment's cells raises DTW_ERR_CUDA (it cannot happen for a
// finite end cell).
constexpr int kWalkWarps = 2;  // fragments per CTA
__global__ void __launch_bounds__(32 * kWalkWarps)
    k_bt_subseq(const WsFrag* __restrict__ fr, int N, const int* __restrict__ ends,
                int32_t* __restrict__ scratch, int* __restrict__ count, DevCtl* ctl) {
    __shared__ uint32_t s_win[kWalkWarps][kWalkWords];
    const int k = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    const int lane = threadIdx.x & 31;
    if (k >= N) return;
    if (ctl->status != 0) {
        if (lane == 0) count[k] = 0;
        return;
    }
    const WsFrag f = fr[k];
    int i = f.len - 1, j = max(ends[k], 0);
    // cell n goes to pair row0 + len - 1 - n
    int2* out = reinterpret_cast<int2*>(scratch) + (f.row0 + f.len - 1);
    WindowWalker w{f.bp, f.nchunk, f.rps, f.wpb, lane, s_win[threadIdx.x >> 5], 0, 0};
    int n = 0, last = -1;  // cells so far, row of the last one
    while (i >= 0 && j >= 0) {
        w.load(i, j);
        int r = w.row(i), c = w.col(j), got;
        do {
            int mr, mc;
            got = w.steps32(r, c, 0, mr, mc);
            if (lane < got) out[-(n + lane)] = make_int2(f.row0 + w.row0 + mr, w.col(mc));
            if (got > 0) last = w.row0 + __shfl_sync(0xffffffffu, mr, got - 1);
            n += got;
        } while (got == 32);
        i = w.row0 + r;
        j = w.col(c);
    }
    const bool bad = last != 0;  // the walk has to end in the fragment's row 0
    if (lane == 0) {
        if (bad) raise_status(ctl, DTW_ERR_CUDA, 22);
        count[k] = bad ? 0 : n;
    }
}

// The fragment paths one after another, one CTA per fragment: fragment k's n_k
// pairs sit at the end of its slots [row0, row0 + len), and go behind those of the
// fragments before it; *path_len = sum n_k (or -status).
__global__ void __launch_bounds__(kCompactThreads)
    k_compact(const WsFrag* __restrict__ fr, int N, const int* __restrict__ count,
              const int32_t* __restrict__ scratch, int32_t* __restrict__ path,
              int* __restrict__ path_len, const DevCtl* ctl) {
    const int st = ctl->status;
    const int k = blockIdx.x;
    if (st != 0) {
        if (k == 0 && threadIdx.x == 0) *path_len = -st;
        return;
    }
    __shared__ int s_before[kCompactThreads / 32];
    int before = 0;
    for (int q = threadIdx.x; q < k; q += blockDim.x) before += count[q];
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) before += __shfl_xor_sync(0xffffffffu, before, off);
    if ((threadIdx.x & 31) == 0) s_before[threadIdx.x >> 5] = before;
    __syncthreads();
    before = 0;
#pragma unroll
    for (int q = 0; q < kCompactThreads / 32; ++q) before += s_before[q];
    const int n = count[k];
    const WsFrag f = fr[k];
    const int32_t* src = scratch + 2 * (size_t)(f.row0 + f.len - n);
    for (int q = threadIdx.x; q < 2 * n; q += blockDim.x) path[2 * (size_t)before + q] = src[q];
    if (k == N - 1 && threadIdx.x == 0) *path_len = before + n;
}

}  // namespace

// Lexicographic (value, column) minimum: the same choice as better() when the
// columns of the two arguments are in order, for any order of arguments.
__device__ __forceinline__ MinArg lex_min(MinArg a, MinArg b) {
    return (b.v < a.v || (b.v == a.v && b.j < a.j)) ? b : a;
}

// Barrier over the CTAs of a cooperative launch (all resident at once):
// bar[0] counts arrivals, bar[1] is the generation the last arrival bumps.
// Bounded: a CTA gives up when the call has failed (any status) or after
// waiting timeout_ns (raising DTW_ERR_TIMEOUT, detail 23), and then returns
// false, as every CTA does once the call has failed.
__device__ __forceinline__ bool grid_barrier(unsigned* bar, DevCtl* ctl, long long timeout_ns) {
    __shared__ int s_ok;
    __syncthreads();
    if (threadIdx.x == 0) {
        int ok = 1;
        const unsigned g = ld_acquire_g(bar + 1);
        __threadfence();
        if (atomicAdd(bar, 1u) == gridDim.x - 1) {
            atomicExch(bar, 0u);
            __threadfence();
            st_release_g(bar + 1, g + 1);
        } else {
            const long long t0 = global_ns();
            while (ld_acquire_g(bar + 1) == g) {
                if (read_status(ctl) != 0) {
                    ok = 0;
                    break;
                }
                if (global_ns() - t0 > timeout_ns) {
                    raise_status(ctl, DTW_ERR_TIMEOUT, 23);
                    ok = 0;
                    break;
                }
                __nanosleep(32);
            }
        }
        s_ok = ok && read_status(ctl) == 0;
    }
    __syncthreads();
    return s_ok;
}

// The whole segment DP in one cooperative launch: one CTA per tile of kTile
// columns, fragments one after another, two bounded grid barriers per
// fragment (the tiles' minima complete; D_seg[k] complete before fragment
// k+1 reads it).  Same values and columns as k_seg_tile + k_seg_fix.
__global__ void __launch_bounds__(kTile)
    k_seg_all(const WsFrag* __restrict__ fr, const float* __restrict__ lastrow, size_t stride,
              int N, int Lb, const int* __restrict__ delta, float* __restrict__ Dseg,
              int* __restrict__ arg, MinArg* __restrict__ agg, unsigned* __restrict__ bar,
              int* __restrict__ ends, float* __restrict__ total, DevCtl* ctl,
              long long timeout_ns) {
    __shared__ MinArg s_warp[32];
    __shared__ MinArg s_carry;
    const int t = blockIdx.x;
    const int j = t * kTile + threadIdx.x;
    // a fragment whose DP failed (a bounded wait expired) fails the call
    if (t == 0 && threadIdx.x == 0)
        for (int q = 0; q < N; ++q) {
            const int st = fr[q].pctl->status;
            if (st != 0) {
                raise_status(ctl, st, 20);
                break;
            }
        }
    MinArg v{INFINITY, -1};
    for (int k = 0; k < N; ++k) {
        const float* cs = lastrow + (size_t)k * stride;
        const float* prev = k > 0 ? Dseg + (size_t)(k - 1) * Lb : nullptr;
        const int dk = k > 0 ? delta[k] : 0;
        v = MinArg{INFINITY, -1};
        if (j < Lb) {
            // D_seg[k-1] was written by other CTAs of this launch: read through L2
            const float m = k == 0 ? cs[j] : (j - dk >= 0 ? __ldcg(prev + j - dk) + cs[j] : INFINITY);
            v = MinArg{attainable(m), j};
        }
        v = block_scan_min(v, s_warp);
        if (threadIdx.x == blockDim.x - 1) {
            volatile MinArg* va = agg;
            va[t].v = v.v;
            va[t].j = v.j;
        }
        if (!grid_barrier(bar, ctl, timeout_ns)) return;
        // the carry into this tile: the minimum over the tiles before it
        if (threadIdx.x < 32) {
            MinArg c{INFINITY, -1};
            const volatile MinArg* va = agg;
            for (int q = threadIdx.x; q < t; q += 32) c = lex_min(c, MinArg{va[q].v, va[q].j});
#pragma unroll
            for (int off = 16; off > 0; off >>= 1) {
                MinArg o;
                o.v = __shfl_xor_sync(0xffffffffu, c.v, off);
                o.j = __shfl_xor_sync(0xffffffffu, c.j, off);
                c = lex_min(c, o);
            }
            if (threadIdx.x == 0) s_carry = c;
        }
        __syncthreads();
        v = better(s_carry, v);
        if (j < Lb) {
            Dseg[(size_t)k * Lb + j] = v.v;
            arg[(size_t)k * Lb + j] = v.j;
        }
        if (!grid_barrier(bar, ctl, timeout_ns)) return;
    }
    // the last fragment's last column: the total and the end frames
    if (j == Lb - 1) {
        if (ctl->status != 0) return;
        if (!(v.v < INFINITY)) {
            raise_status(ctl, DTW_ERR_UNREACHABLE, 21);
            return;
        }
        *total = v.v;
        int e = v.j;
        ends[N - 1] = e;
        for (int q = N - 1; q > 0; --q) {
            e = __ldcg(arg + (size_t)(q - 1) * Lb + (e - delta[q]));
            ends[q - 1] = e;
        }
    }
}

// The whole segment DP in one thread-block cluster, for a B of up to 131072
// columns: CTA r has the columns [r kCols, (r + 1) kCols) and keeps their D_seg in
// shared memory, where the next fragment's matches read it, from the CTAs to the
// left where delta reaches that far.  What bounds it is the chain of fragments, each
// two exchanges long (the CTAs' minima; D_seg before fragment k+1 reads it): a
// barrier of the grid costs a round trip through L2 and its poll, one of the cluster
// less than half of that, and eight SMs hold the columns of a few minutes to an hour
// of frames.  A thread loads and stores columns kSegThreads apart, and scans
// kPer neighbouring ones (shared memory, one word of padding in 32, no bank
// conflicts).  Same values and columns as k_seg_tile + k_seg_fix.  32 fragments x
// 50021 columns: 140 us, 248 with k_seg_all (the whole call 4.40 -> 4.28 ms).
constexpr int kSegThreads = 1024;
__device__ __forceinline__ int seg_slot(int p) { return p + (p >> 5); }
template <int kPer>
constexpr int seg_smem() {
    return 2 * (kSegThreads * kPer + kSegThreads * kPer / 32) * (int)sizeof(float);
}

template <int kPer>
__global__ void __launch_bounds__(kSegThreads)
    k_seg_cluster(const WsFrag* __restrict__ fr, const float* __restrict__ lastrow, size_t stride,
                  int N, int Lb, const int* __restrict__ delta, int* arg, int* ends, float* total,
                  DevCtl* ctl) {
    constexpr int kCols = kSegThreads * kPer;
    extern __shared__ float s_seg[];
    float* Ds = s_seg;                              // D_seg of the fragment before
    float* Ms = s_seg + kCols + kCols / 32;         // its matches, then its arg
    __shared__ MinArg s_warp[kSegThreads / 32], s_cta[8];
    __shared__ int s_bad;
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    const unsigned rank = cluster_rank(), cn = cluster_size();
    const int c0 = (int)rank * kCols;
    const unsigned ds = smem_u32(Ds);
    // a fragment whose DP failed (a bounded wait expired) fails the call
    if (rank == 0) {
        if (tid == 0) s_bad = N;
        __syncthreads();
        for (int q = tid; q < N; q += kSegThreads)
            if (fr[q].pctl->status != 0) atomicMin(&s_bad, q);
        __syncthreads();
        if (tid == 0 && s_bad < N) raise_status(ctl, fr[s_bad].pctl->status, 20);
    }
    float cs[kPer];  // C_seg of fragment k at columns c0 + tid + i kSegThreads
    auto load = [&](int k) {
#pragma unroll
        for (int i = 0; i < kPer; ++i) {
            const int col = c0 + tid + i * kSegThreads;
            cs[i] = col < Lb ? lastrow[(size_t)k * stride + col] : INFINITY;
        }
    };
    load(0);
    cluster_sync_all();  // every CTA runs before any is stored into
    for (int k = 0; k < N; ++k) {
        const int dk = k > 0 ? delta[k] : 0;
        float m[kPer];
#pragma unroll
        for (int i = 0; i < kPer; ++i) {
            const int src = c0 + tid + i * kSegThreads - dk;
            m[i] = k == 0 ? 0.f : INFINITY;
            if (k > 0 && src >= 0)
                m[i] = ld_cluster_f32(map_rank(ds + 4u * (unsigned)seg_slot(src % kCols), src / kCols));
        }
#pragma unroll
        for (int i = 0; i < kPer; ++i)
            Ms[seg_slot(tid + i * kSegThreads)] = attainable(k == 0 ? cs[i] : m[i] + cs[i]);
        if (k + 1 < N) load(k + 1);
        __syncthreads();
        // the minimum of the thread's columns, of the lanes and warps before it
        MinArg x{INFINITY, -1};
#pragma unroll
        for (int i = 0; i < kPer; ++i)
            x = better(x, MinArg{Ms[seg_slot(tid * kPer + i)], c0 + tid * kPer + i});
#pragma unroll
        for (int off = 1; off < 32; off <<= 1) {
            MinArg o;
            o.v = __shfl_up_sync(0xffffffffu, x.v, off);
            o.j = __shfl_up_sync(0xffffffffu, x.j, off);
            if (lane >= off) x = better(o, x);
        }
        if (lane == 31) s_warp[w] = x;
        MinArg run;
        run.v = __shfl_up_sync(0xffffffffu, x.v, 1);
        run.j = __shfl_up_sync(0xffffffffu, x.j, 1);
        if (lane == 0) run = MinArg{INFINITY, -1};
        __syncthreads();
        MinArg c = lane < w ? s_warp[lane] : MinArg{INFINITY, -1};
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) {
            MinArg o;
            o.v = __shfl_xor_sync(0xffffffffu, c.v, off);
            o.j = __shfl_xor_sync(0xffffffffu, c.j, off);
            c = lex_min(c, o);
        }
        if (w == kSegThreads / 32 - 1) {  // the CTA's minimum, to every CTA
            const MinArg all = better(c, s_warp[w]);
            if (lane < (int)cn) {
                const unsigned at = map_rank(smem_u32(&s_cta[rank]), (unsigned)lane);
                st_cluster_u32(at, __float_as_uint(all.v));
                st_cluster_u32(at + 4, (unsigned)all.j);
            }
        }
        run = better(c, run);
        cluster_sync_all();
        c = MinArg{INFINITY, -1};
        for (unsigned r = 0; r < rank; ++r) c = better(c, s_cta[r]);
        run = better(c, run);
#pragma unroll
        for (int i = 0; i < kPer; ++i) {
            const int p = seg_slot(tid * kPer + i);
            run = better(run, MinArg{Ms[p], c0 + tid * kPer + i});
            Ds[p] = run.v;
            Ms[p] = __int_as_float(run.j);
        }
        cluster_sync_all();
        // (the same thread stores the next fragment's matches there)
#pragma unroll
        for (int i = 0; i < kPer; ++i) {
            const int p = tid + i * kSegThreads;
            if (c0 + p < Lb) arg[(size_t)k * Lb + c0 + p] = __float_as_int(Ms[seg_slot(p)]);
        }
    }
    // the last fragment's last column: the total and the end frames
    const int last = Lb - 1 - c0;
    if (tid == 0 && last >= 0 && last < kCols) {
        if (read_status(ctl) != 0) return;
        const float v = Ds[seg_slot(last)];
        if (!(v < INFINITY)) {
            raise_status(ctl, DTW_ERR_UNREACHABLE, 21);
            return;
        }
        *total = v;
        int e = __float_as_int(Ms[seg_slot(last)]);
        ends[N - 1] = e;
        for (int q = N - 1; q > 0; --q) {
            e = __ldcg(arg + (size_t)(q - 1) * Lb + (e - delta[q]));
            ends[q - 1] = e;
        }
    }
}

template <int kPer>
cudaError_t launch_seg_cluster(const WsFrag* fr, const float* lastrow, size_t stride, int N, int Lb,
                               const int* delta, int* arg, int* ends, float* total, DevCtl* ctl,
                               cudaStream_t s) {
    static DeviceSlots done;
    cudaError_t e = raise_smem_once(k_seg_cluster<kPer>, seg_smem<kPer>(), done);
    if (e != cudaSuccess) return e;
    const int cn = (Lb + kSegThreads * kPer - 1) / (kSegThreads * kPer);
    cudaLaunchAttribute at = {};
    at.id = cudaLaunchAttributeClusterDimension;
    at.val.clusterDim.x = (unsigned)cn;
    at.val.clusterDim.y = 1;
    at.val.clusterDim.z = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)cn);
    cfg.blockDim = dim3(kSegThreads);
    cfg.dynamicSmemBytes = (size_t)seg_smem<kPer>();
    cfg.stream = s;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, k_seg_cluster<kPer>, fr, lastrow, stride, N, Lb, delta, arg,
                              ends, total, ctl);
}

cudaError_t launch_seg_dp(const WsFrag* fr, const float* lastrow, size_t stride, int N, int Lb,
                          const int* delta, float* Dseg, int* arg, void* agg, unsigned* done,
                          int* ends, float* total, DevCtl* ctl, long long timeout_ns,
                          cudaStream_t s) {
    // one cluster where its eight CTAs hold the columns (131072 of them)
    cudaError_t e = cudaErrorInvalidValue;
    const int per = (Lb + 8 * kSegThreads - 1) / (8 * kSegThreads);
    if (per <= 4)
        e = launch_seg_cluster<4>(fr, lastrow, stride, N, Lb, delta, arg, ends, total, ctl, s);
    else if (per <= 8)
        e = launch_seg_cluster<8>(fr, lastrow, stride, N, Lb, delta, arg, ends, total, ctl, s);
    else if (per <= 16)
        e = launch_seg_cluster<16>(fr, lastrow, stride, N, Lb, delta, arg, ends, total, ctl, s);
    if (e == cudaSuccess) return e;
    (void)cudaGetLastError();
    const int ntile = (Lb + kTile - 1) / kTile;
    e = cudaMemsetAsync(done, 0, 2 * sizeof(unsigned), s);
    if (e != cudaSuccess) return e;
    // one cooperative launch when every tile's CTA can be resident at once
    // (CTAs resident on the current device, looked up once per device)
    constexpr int kMaxDev = 64;
    static std::atomic<int> resident_of[kMaxDev];  // 0 = not looked up yet, else 1 + count
    int dev = 0, resident = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) {
        (void)cudaGetLastError();
        dev = -1;
    }
    if (dev >= 0 && dev < kMaxDev && resident_of[dev].load() > 0) {
        resident = resident_of[dev].load() - 1;
    } else if (dev >= 0) {
        int sms = 0, per_sm = 0;
        if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
            cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_seg_all, kTile, 0) !=
                cudaSuccess) {
            (void)cudaGetLastError();
        } else {
            resident = sms * per_sm;
            if (dev < kMaxDev) resident_of[dev].store(resident + 1);
        }
    }
    if (ntile <= resident) {
        MinArg* aggp = static_cast<MinArg*>(agg);
        void* args[] = {(void*)&fr,   (void*)&lastrow, (void*)&stride, (void*)&N,
                        (void*)&Lb,   (void*)&delta,   (void*)&Dseg,   (void*)&arg,
                        (void*)&aggp, (void*)&done,    (void*)&ends,   (void*)&total,
                        (void*)&ctl,  (void*)&timeout_ns};
        return cudaLaunchCooperativeKernel((const void*)k_seg_all, dim3(ntile), dim3(kTile), args,
                                           0, s);
    }
    for (int k = 0; k < N && e == cudaSuccess; ++k) {
        k_seg_tile<<<ntile, kTile, 0, s>>>(fr, lastrow, stride, N, Lb, k, delta, Dseg,
                                           static_cast<MinArg*>(agg), done, ctl);
        k_seg_fix<<<ntile, kTile, 0, s>>>(lastrow, stride, N, Lb, k, delta, Dseg, arg,
                                          static_cast<const MinArg*>(agg), ends, total, ctl);
        e = cudaGetLastError();
    }
    return e;
}

size_t seg_dp_scratch_bytes(int Lb) { return sizeof(MinArg) * (size_t)((Lb + kTile - 1) / kTile); }

cudaError_t launch_bt_subseq(const WsFrag* fr, int N, const int* ends, int32_t* scratch,
                             int* count, int32_t* path, int* path_len, DevCtl* ctl,
                             cudaStream_t s) {
    k_bt_subseq<<<(N + kWalkWarps - 1) / kWalkWarps, 32 * kWalkWarps, 0, s>>>(fr, N, ends, scratch,
                                                                               count, ctl);
    k_compact<<<N, kCompactThreads, 0, s>>>(fr, N, count, scratch, path, path_len, ctl);
    return cudaGetLastError();
}

}  // namespace pardtw

// Launch of the warp-pair DP of one pair in thread-block clusters
// (k_dp_split<..., kCl = true>, see dp_split.cuh), shared by the translation
// units that instantiate it (dp_split_cl.cu for D <= 32 and the BF16 cost,
// dp_split_wide.cu for the FP32 cost at D = 64, 128).
//
// Between two CTAs the strip border otherwise goes through global memory:
// the writer warp of the CTA above stores it, the reader warp of the CTA
// below polls it.  In a cluster the writer warp stores it straight into the
// slots of the CTA below, so only one hop in cn stays global.  From strip to
// strip of a 4000-column chain at D = 12, two strips a CTA: 1.55 us without
// clusters, 0.75 in them (one strip a CTA: 2.4 and 0.9), of which the 31 lanes'
// skew alone is 0.66.
//
// Every CTA of a cluster sits on an SM of its own (the dynamic shared
// memory is raised so that two CTAs cannot share an SM, which would put two
// DP warps on one SM sub-partition).  One strip a CTA where one or two cost
// warps cannot keep up with a DP warp (D > 16, the BF16 cost: three or four cost
// warps a strip, on the sub-partitions beside the DP warp's), else two.  The
// cluster size: see launch_cl.  Measured (DP, ms): 20000 x 25000, D = 12, clusters
// of 8 / 6 / 4 / 2: 0.906 / 0.916 / 0.928 / 0.976; 100000 x 126231 (335 groups active
// at once, 152 SMs): 6.87 / 6.38 / 6.19 / 5.88; 40000 x 48000, D = 128, BF16: 2.59 / 2.48
// / 2.46 / 2.45 with one strip a CTA, 3.16 without clusters and two.
#pragma once
#include <algorithm>
#include <mutex>

#include "dp_split.cuh"

namespace pardtw {
namespace {

constexpr int kClSmemFloor = 120 * 1024;  // > half an SM's shared memory: one CTA per SM
constexpr int kClMaxDev = 64;
constexpr int kNClSizes = 7;
constexpr int kClSizes[kNClSizes] = {8, 7, 6, 5, 4, 3, 2};

template <int DP, bool kBF, bool kT, int NS = 2>
struct ClKernel {
    static constexpr int R = 3;
    static constexpr int kThreads = split_threads<DP, NS, kBF>();
    static constexpr auto kern() { return k_dp_split<DP, R, NS, false, kBF, false, kT, true>; }
    static int smem() {
        return std::max(NS * SplitSmem<DP, R, NS, kBF, true>::kStripBytes, kClSmemFloor);
    }
};

struct ClInfo {
    bool ready = false, ok = false;
    int max_clusters[kNClSizes] = {};  // resident clusters of size kClSizes[k]
};

cudaLaunchConfig_t cl_config(dim3 grid, int threads, int smem, cudaStream_t s,
                             cudaLaunchAttribute* at, int cn) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = dim3((unsigned)threads);
    cfg.dynamicSmemBytes = (size_t)smem;
    cfg.stream = s;
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = (unsigned)cn;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    at[1] = chained_attr(true);
    cfg.attrs = at;
    cfg.numAttrs = 2;
    return cfg;
}

// Attributes and cluster occupancy of one instantiation, once per device.
template <int DP, bool kBF, bool kT, int NS>
const ClInfo& cl_info(int dev) {
    static ClInfo info[kClMaxDev];
    static std::mutex mu;
    using K = ClKernel<DP, kBF, kT, NS>;
    std::lock_guard<std::mutex> lock(mu);
    ClInfo& ci = info[dev];
    if (ci.ready) return ci;
    ci.ready = true;
    auto* kern = K::kern();
    if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, K::smem()) !=
        cudaSuccess) {
        (void)cudaGetLastError();
        return ci;
    }
    for (int k = 0; k < kNClSizes; ++k) {
        cudaLaunchAttribute at[2];
        cudaLaunchConfig_t cfg =
            cl_config(dim3((unsigned)kClSizes[k]), K::kThreads, K::smem(), nullptr, at, kClSizes[k]);
        int n = 0;
        if (cudaOccupancyMaxActiveClusters(&n, kern, &cfg) != cudaSuccess) {
            (void)cudaGetLastError();
            n = 0;
        }
        ci.max_clusters[k] = n;
    }
    ci.ok = true;
    return ci;
}

// Strips of `a` that are active at once: those whose rows a path can cross at
// one column (the most at the corners of the path region); a band's strips are
// short and follow one another, so few are.
inline int peak_strips(const DpArgs& a) {
    if (a.ranges) return 1;
    const long long r = a.La, c = a.Lb;
    long long most = 0;
    for (const long long col : {(2 * r - c) / 3, (4 * c - 2 * r) / 3}) {
        const long long lo = std::max(col / 2, r - 2 * (c - col));
        const long long hi = std::min(2 * col, r - (c - col) / 2);
        most = std::max(most, std::min(hi, r) - std::max(lo, 0LL));
    }
    return (int)(most / a.rps) + 1;
}

template <int DP, bool kBF, bool kT, int NS = 2>
cudaError_t launch_cl(const DpArgs& pair, cudaStream_t s, bool* used) {
    *used = false;
    DpArgs a = pair;
    a.ngroups = (a.nstrips + NS - 1) / NS;
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kClMaxDev) {
        (void)cudaGetLastError();
        return cudaSuccess;
    }
    const ClInfo& ci = cl_info<DP, kBF, kT, NS>(dev);
    if (!ci.ok) return cudaSuccess;
    // the largest clusters (fewest hops through global memory) of which enough
    // are resident for the groups that are active at once, else those that hold
    // the most groups
    const int need = std::min(a.ngroups, (peak_strips(a) + NS - 1) / NS);
    int cn = 0, nclusters = 0;
    for (int k = 0; k < kNClSizes; ++k) {
        if (ci.max_clusters[k] <= 0) continue;
        cn = kClSizes[k];
        nclusters = std::min(ci.max_clusters[k], (a.ngroups + cn - 1) / cn);
        if (ci.max_clusters[k] * cn >= need) break;
    }
    if (cn == 0) return cudaSuccess;
    using K = ClKernel<DP, kBF, kT, NS>;
    cudaLaunchAttribute at[2];
    cudaLaunchConfig_t cfg =
        cl_config(dim3((unsigned)(nclusters * cn)), K::kThreads, K::smem(), s, at, cn);
    const cudaError_t e = cudaLaunchKernelEx(&cfg, K::kern(), a,
                                             static_cast<const DpArgs*>(nullptr),
                                             static_cast<const int2*>(nullptr), 0,
                                             static_cast<int*>(nullptr));
    if (e == cudaSuccess) *used = true;
    return e;
}

}  // namespace
}  // namespace pardtw

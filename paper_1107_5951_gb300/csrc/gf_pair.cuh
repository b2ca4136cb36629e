// gf_pair.cuh -- pieces shared by the direct sums: the FP64 kernel value
// m / r^3, compensated running sums, and the split of one observer tile's
// sources over the warps of a thread-block cluster.
//
// A direct sum of M observers over N sources has M independent outputs, and
// surveys of a few hundred to a few thousand stations leave most of the chip
// idle when one thread walks all N sources of its observer (16^3 voxels with
// a 2x2x2 rule at 4096 stations: 16 blocks of 256 threads, 41.6 ms).  Here a
// tile is 32 or 64 observers (one or two per lane); every warp of every block
// of a cluster takes a share of the sources for the whole tile, and the
// partial sums meet in shared memory (the block's 8 warps) and then over the
// cluster's distributed shared memory, in a fixed order: no workspace, and
// the same result on every run.  Few sources over many observers need no sharing, and
// adding up the shares would take longer than the sums: there a warp takes a tile by
// itself (kSolo; pair_cluster chooses).
#pragma once

#include <cooperative_groups.h>

#include <algorithm>

#include "gf_internal.cuh"

namespace gf {
namespace {

constexpr int kPairWarps = 8;
constexpr int kPairThreads = kPairWarps * 32;
constexpr int kPairMaxCluster = 8;   // the portable cluster size

// m r2^(-3/2) for normal finite r2, 0 otherwise (a source on the observer, or
// beyond the range of doubles).  The FP64 pipe does two instructions a
// clock and SM here, so it is what bounds an FP64 pair; the integer and
// special-function units are free beside it.  The seed y0 = (r2)^(-1/2) to
// FP32 comes from the special-function unit (r2 = 4^s f, f in [1, 4), by
// exponent arithmetic), and with e = 1 - r2 y0^2 (|e| < 2^-20)
//   r2^(-3/2) = y0^3 (1 - e)^(-3/2) = y0^3 (1 + 3/2 e + 15/8 e^2 + O(e^3)),
// the binomial series cut where its terms fall below 2^-60: 7 FP64
// instructions, against 9 for a rounded reciprocal square root and its cube.
__device__ __forceinline__ double inv_r3(double r2, double m) {
    const unsigned hi = (unsigned)__double2hiint(r2), lo = (unsigned)__double2loint(r2);
    const int ex = (int)(hi >> 20) - 1023;   // unbiased exponent (sign bit clear)
    const float f = __uint_as_float(((unsigned)(127 + (ex & 1)) << 23) | ((hi & 0xfffffu) << 3) | (lo >> 29));
    float y;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(f));
    const unsigned yb = __float_as_uint(y);
    // y 2^-s as a double, s = floor(ex / 2)
    const int ey = (int)(yb >> 23) - 127 - (ex >> 1) + 1023;
    const double y0 = __hiloint2double((int)(((unsigned)ey << 20) | ((yb >> 3) & 0xfffffu)), (int)(yb << 29));
    const double s = y0 * y0;
    const double e = fma(-r2, s, 1.0);
    const double wm = (s * y0) * m;
    const double q = fma(fma(1.875, e, 1.5), e, 1.0);
    const double k = wm * q;
    return (hi - 0x00100000u) < 0x7fe00000u ? k : 0.0;
}

__device__ __forceinline__ void two_sum_d(double &hi, double &lo, double x) {
    const double s = hi + x;
    const double bp = s - hi;
    lo += (hi - (s - bp)) + (x - bp);
    hi = s;
}

// Sums (s[v], c[v]) over the block's warps and the cluster's blocks, in
// warp and rank order.  sh: [kPairWarps + 1][NV * 32] double2 of shared
// memory.  Returns, in every thread t < NV * 32 of rank 0, the total of
// value t / 32 of lane t % 32 (high part + compensation); 0 elsewhere.
// All threads of the cluster call it.
template <int NV>
__device__ __forceinline__ double cluster_total(const double (&s)[NV], const double (&c)[NV], double2 *sh) {
    namespace cg = cooperative_groups;
    static_assert(NV * 32 <= kPairThreads, "one thread per value and lane");
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    double2 *part = sh + kPairWarps * NV * 32;
#pragma unroll
    for (int v = 0; v < NV; ++v) sh[(warp * NV + v) * 32 + lane] = make_double2(s[v], c[v]);
    __syncthreads();
    const int t = threadIdx.x;
    if (t < NV * 32) {
        double S = 0.0, C = 0.0;
#pragma unroll
        for (int w = 0; w < kPairWarps; ++w) {
            const double2 p = sh[w * NV * 32 + t];
            two_sum_d(S, C, p.x);
            C += p.y;
        }
        part[t] = make_double2(S, C);
    }
    cg::cluster_group cl = cg::this_cluster();
    cl.sync();
    double out = 0.0;
    if (cl.block_rank() == 0 && t < NV * 32) {
        double S = 0.0, C = 0.0;
        for (unsigned r = 0; r < cl.num_blocks(); ++r) {
            const double2 p = *cl.map_shared_rank(part + t, r);
            two_sum_d(S, C, p.x);
            C += p.y;
        }
        out = S + C;
    }
    cl.sync();   // no block leaves while another may read its sums
    return out;
}

template <int NV>
constexpr size_t pair_smem() {
    return sizeof(double2) * (kPairWarps + 1) * NV * 32;
}

// How one SM's time goes in a direct sum, in microseconds: a work unit of one tile,
// a block's start and its cluster_total, and how much longer a warp alone on an SM
// takes over a unit than warps that fill it take on average.
struct PairCost {
    double unit, block, alone;
};

// Blocks per cluster for `tiles` observer tiles and `units` work units per tile, or
// 0: a warp alone to a tile, without partial sums to add up.  The size with the
// least time for the SM with the most blocks (the smaller size when it is within 2%
// of the best), with at least two units for each warp of a cluster.  A tile's
// cluster_total is some 400 FP64 instructions, 5 to 8 us of an SM.  A million observers
// of one voxel 557 us (mixed) and 868 (FP64) with it, 40 and 108 a warp to a tile (a
// thread per observer before either: 38 and 103); of 4^3 voxels 617 and 2,405, now 74
// and 1,753 (82 and 2,179); of 8^3 882, now 285 (515), FP64 12.6 ms (17.0).  The size
// decides how an observer's sum associates: callers count the tiles of one batch
// member, so that a member's sums are the same bits alone and in any batch.  *time:
// the SM's time, in microseconds.
inline int pair_cluster(int64_t tiles, int64_t units, PairCost cost, double *time = nullptr) {
    const int64_t sms = sm_count();
    const int64_t most = std::max<int64_t>(1, std::min<int64_t>(kPairMaxCluster, units / (2 * kPairWarps)));
    // a warp to a tile (a tenth slower a unit than warps that share a block)
    double best_us = 1.1 * (double)units * cost.unit * std::max((double)((tiles + sms - 1) / sms), cost.alone);
    int best = 0;
    for (int64_t c = 1; c <= most; ++c) {
        const int64_t rounds = (tiles * c + sms - 1) / sms;
        // the warps of a block that have no unit do not help
        const double share = std::max(1.0 / (double)c, cost.alone / (double)std::max<int64_t>(1, units));
        const double us = (double)rounds * (cost.block + (double)units * cost.unit * share);
        if (us < 0.98 * best_us) {
            best_us = us;
            best = (int)c;
        }
    }
    if (time) *time = best_us;
    return best;
}

// Launch of `kernel` on tiles x batch warps.
template <class... A, class... B>
gf_status pair_launch_solo(void (*kernel)(A...), int64_t tiles, int batch, cudaStream_t st, B &&...args) {
    kernel<<<dim3((unsigned)tiles, (unsigned)batch), 32, 0, st>>>(std::forward<B>(args)...);
    GF_KERNEL_DONE();
    return GF_OK;
}

// Launch of `kernel` on tiles x batch clusters of `cluster` blocks.
template <class... A, class... B>
gf_status pair_launch(void (*kernel)(A...), int64_t tiles, int batch, int cluster, cudaStream_t st, B &&...args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(tiles * cluster), (unsigned)batch);
    cfg.blockDim = dim3(kPairThreads);
    cfg.stream = st;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = (unsigned)cluster;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    GF_CUDA(cudaLaunchKernelEx(&cfg, kernel, std::forward<B>(args)...));
    GF_KERNEL_DONE();
    return GF_OK;
}

}  // namespace
}  // namespace gf

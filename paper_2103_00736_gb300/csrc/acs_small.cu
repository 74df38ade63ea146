// The iteration kernel of small problems: one thread-block cluster.
//
// A problem of a few hundred constraints with the cached projection operator
// does 1e4 to 1e6 FP64 multiply-adds an iteration in four phases; on the whole
// grid its time is the grid barriers (2 us each, 4 with a reduction) and the
// instructions that 152 x 32 mostly idle warps spend around them (16 % of them
// spills of the 64-register build).  On one cluster the barrier is the hardware's,
// partials travel through distributed shared memory, and 512 threads a CTA have
// 128 registers each, so nothing spills.  The FP64 pipe then sets the limit: 2 multiply-adds per clock per SM
// on 16 SMs instead of 152, hence the size rule in small_cluster().
#include <cuda_runtime.h>

#include "acs_device.cuh"

namespace acs {
namespace {

__global__ void __launch_bounds__(kSmallThreads, 1) small_iter_kernel(const __grid_constant__ IterParams<double> P) {
    if (ld_volatile_int(&P.ctl->status) != ST_RUNNING) return;
    team_set(blockIdx.x, gridDim.x, &P.ctl->bar_count64, P.partials, P.dM, P.dX, 1);
    sync_init(P.ctl->bar_gen);
    cluster_sync();                                      // every CTA's shared memory is in use from here
    solve_loop<double>(stage_params(P), ST_RUNNING);
    cluster_sync();                                      // no CTA leaves while its shared memory may be written
}

}  // namespace

// CTAs of the one-cluster launch for this problem, 0 for the whole grid.  The
// line: multiply-adds of an iteration, m^2 for the cached operator and the
// stored entries of A and A' once each.  Measured, us an iteration (and the
// factorisation's ms), cluster against grid: sparse LP m = 200 19.0 (0.56) /
// 28.1 (0.58), m = 400 25.9 (1.4) / 31.3 (1.0), m = 512 27.6 (2.1) / 31.2
// (1.25: at 100 iterations a factorisation the grid is ahead), m = 700 37.7 /
// 32.5; dense SOCP m = 200 36.5 / 48.8, m = 296 53.9 / 56.7, m = 400 69 / 61.
// Coordinates and cones cost too: at two rounds of them the grid is ahead for sparse
// rows (m = 200 with 2 entries a column: n = 10000 27.8 / 25.7, n = 20000 34.3 / 27.2,
// n = 40000 50.7 / 30.8; two full rows the other way, n = 20000 88 / 114), and a wider
// problem is left to it.
int small_cluster(const Problem* P) {
    if (P->dense != 1) return 0;
    const double work = (double)P->m * P->m + (double)P->padded_A + (double)P->padded_AT;
    if (work > 2.5e5) return 0;
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeClusterDimension;
    at.val.clusterDim.y = at.val.clusterDim.z = 1;
    if (cudaFuncSetAttribute(small_iter_kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess) {
        cudaGetLastError();
        return 0;
    }
    for (int c = kMaxCluster; c >= 8; c /= 2) {
        if (P->n > 2 * c * kSmallThreads) return 0;
        cudaLaunchConfig_t cfg{};
        cfg.gridDim = dim3(c);
        cfg.blockDim = dim3(kSmallThreads);
        cfg.attrs = &at;
        cfg.numAttrs = 1;
        at.val.clusterDim.x = c;
        int n = 0;
        if (cudaOccupancyMaxActiveClusters(&n, small_iter_kernel, &cfg) == cudaSuccess && n >= 1) return c;
        cudaGetLastError();
    }
    return 0;
}

cudaError_t launch_small(const IterParams<double>& Q, int ctas, cudaStream_t stream) {
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeClusterDimension;
    at.val.clusterDim.x = ctas;
    at.val.clusterDim.y = at.val.clusterDim.z = 1;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(ctas);
    cfg.blockDim = dim3(kSmallThreads);
    cfg.stream = stream;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, small_iter_kernel, Q);
}

}  // namespace acs

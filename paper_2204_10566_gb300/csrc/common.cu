// Precision-independent kernels: the fixed-order final pass of the FP64
// health reduction and the time-average readback.
#include <algorithm>
#include <cstdlib>

#include "lbm_internal.h"

namespace lbm {

int barrier_polls() {
    const char *s = std::getenv("LBM_BARRIER_POLLS");
    return s ? std::max(0, std::atoi(s)) : 1 << 22;
}

int cooperative_blocks(int blocks) {
    const char *s = std::getenv("LBM_COOPERATIVE_BLOCKS");
    return s && blocks > 0 ? std::max(1, std::atoi(s)) : blocks;
}

bool launch_refused(cudaError_t e) {
    return e == cudaErrorCooperativeLaunchTooLarge || e == cudaErrorNotSupported || e == cudaErrorLaunchOutOfResources;
}

int fluid_blocks(int32_t nchunks) {
    const int64_t threads = (int64_t)nchunks * CHUNK;
    return (int)((threads + STEP_THREADS - 1) / STEP_THREADS);
}

// Enough blocks to fill the device; a block's slots follow from this count
// alone, so the totals stay bitwise reproducible.
int reduce_blocks(int64_t nslots) { return (int)std::min<int64_t>((nslots + STEP_THREADS - 1) / STEP_THREADS, 152 * 12); }

int node_blocks(int64_t n) { return (int)((n + STEP_THREADS - 1) / STEP_THREADS); }

// One block sums the per-block partials in a fixed order (each thread a
// fixed strided subset, then a fixed tree), so the totals are bitwise
// reproducible for a given lattice.  health: mass, momentum (3), max |u|,
// non-finite count.  A non-finite count > 0 raises bit 0 of *status.
__global__ void __launch_bounds__(256) k_finalize(const double *partials, int nblocks, double *health,
                                                  uint32_t *status) {
    __shared__ double sh[256][6];
    double r[6] = {0, 0, 0, 0, 0, 0};
    for (int b = threadIdx.x; b < nblocks; b += 256) {
        const double *p = partials + (size_t)b * REDUCE_SLOTS;
#pragma unroll
        for (int k = 0; k < 6; ++k) r[k] = (k == 4) ? fmax(r[k], p[k]) : r[k] + p[k];
    }
#pragma unroll
    for (int k = 0; k < 6; ++k) sh[threadIdx.x][k] = r[k];
    __syncthreads();
    for (int h = 128; h > 0; h >>= 1) {
        if ((int)threadIdx.x < h) {
#pragma unroll
            for (int k = 0; k < 6; ++k)
                sh[threadIdx.x][k] = (k == 4) ? fmax(sh[threadIdx.x][k], sh[threadIdx.x + h][k])
                                              : sh[threadIdx.x][k] + sh[threadIdx.x + h][k];
        }
        __syncthreads();
    }
    if (threadIdx.x == 0) {
#pragma unroll
        for (int k = 0; k < 6; ++k) health[k] = sh[0][k];
        if (sh[0][5] > 0.0) *status |= 1u;
    }
}

cudaError_t launch_finalize(const double *partials, int nblocks, double *health, uint32_t *status,
                            cudaStream_t s) {
    k_finalize<<<1, 256, 0, s>>>(partials, nblocks, health, status);
    return cudaGetLastError();
}

__global__ void k_stats_mean(const double *stats, int ncomp, const int32_t *act, int64_t stride, double inv_n,
                             double *out, double *out2) {
    const int64_t slot = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (slot >= stride) return;
    const int64_t k = act[slot];
    if (k < 0) return;
    if (out2) {
        out[k] = stats[slot] * inv_n;
        out2[k] = stats[stride + slot] * inv_n;
        return;
    }
    for (int q = 0; q < ncomp; ++q) out[(int64_t)ncomp * k + q] = stats[(int64_t)q * stride + slot] * inv_n;
}

cudaError_t launch_stats_mean(const double *stats, int ncomp, const int32_t *act, int64_t stride, double inv_n,
                              double *out, double *out2, cudaStream_t s) {
    k_stats_mean<<<(unsigned)((stride + 255) / 256), 256, 0, s>>>(stats, ncomp, act, stride, inv_n, out, out2);
    return cudaGetLastError();
}

}  // namespace lbm

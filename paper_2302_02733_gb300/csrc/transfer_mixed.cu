// Mixed form of the transfer kernel: the FP64 geodesic path is read back, and the plasma
// fetch, coefficients and transfer run in float.
#include <algorithm>

#include "transfer_kernel.cuh"

namespace prt {
template <int CM, bool JOBS>
static void launch_two(const XferArgs &a, int grid, cudaStream_t s) {
    cudaMemsetAsync(&a.ctr->chain_next, 0, sizeof(unsigned long long), s);
    constexpr int T = PointsCfg<float>::threads;
    // grid counts blocks of kXferThreads
    points_kernel<float, CM, JOBS><<<ray_grid((grid * kXferThreads + T - 1) / T, a.nrays, T / 32), T, 0, s>>>(a);
    chain_kernel<float, float, JOBS><<<ray_grid(2 * grid, a.nrays, kXferThreads), kXferThreads, 0, s>>>(a);
}
void launch_transfer_mixed(const XferArgs &a, int coef, int grid, cudaStream_t s) {
    switch (coef) {
        case 0:
            if (a.jobs)
                launch_two<0, true>(a, grid, s);
            else
                launch_two<0, false>(a, grid, s);
            break;
        case 1: launch_two<1, false>(a, grid, s); break;
        case 2: launch_two<2, false>(a, grid, s); break;
        default: break;
    }
}
void launch_transfer_staged(const XferArgs &a, const CUtensorMap &map, int grid, cudaStream_t s) {
    grid = ray_grid(grid, a.nrays, kXferThreads);
    transfer_kernel_staged<0><<<grid, kXferThreads, 0, s>>>(a, map);
}
int transfer_blocks_per_sm_staged() {
    int n = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, transfer_kernel_staged<0>, kXferThreads, 0) != cudaSuccess) n = 1;
    return n > 0 ? n : 1;
}
void launch_unpol(const XferArgs &a, int grid, cudaStream_t s) {
    grid = ray_grid(grid, a.nrays, kXferThreads / 32);
    if (a.jobs)
        unpol_kernel<float, true><<<grid, kXferThreads, 0, s>>>(a);
    else
        unpol_kernel<float><<<grid, kXferThreads, 0, s>>>(a);
}
void launch_sur_features(const XferArgs &a, int grid, cudaStream_t s) {
    grid = ray_grid(grid, a.nrays, kXferThreads / 32);
    sur_features_pass<float><<<grid, kXferThreads, 0, s>>>(a);
}
static int func_regs(const void *f) {
    cudaFuncAttributes a{};
    if (cudaFuncGetAttributes(&a, f) != cudaSuccess) {
        cudaGetLastError();
        return 255;
    }
    return a.numRegs;
}
int transfer_regs_mixed() {
    int r = func_regs((const void *)points_kernel<float, 0>);
    r = std::max(r, func_regs((const void *)points_kernel<float, 0, true>));
    r = std::max(r, func_regs((const void *)transfer_kernel_staged<0>));
    r = std::max(r, func_regs((const void *)unpol_kernel<float>));
    return std::max(r, func_regs((const void *)unpol_kernel<float, true>));
}
int transfer_blocks_per_sm_mixed() {
    int n = 0;
    constexpr int T = PointsCfg<float>::threads;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, points_kernel<float>, T, 0) != cudaSuccess) n = 1;
    return n > 0 ? n * (T / kXferThreads) : 1;
}
}  // namespace prt

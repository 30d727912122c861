// The kernels' 6x6 solve on systems given as such, one warp each: tests/test_gpu_block_solve.py builds and loads it.
#include "../paper_2101_00585_gb300/csrc/common.cuh"

namespace upslam {
// sys[n][27]: upper triangle of A, b.  xi[n][6], ok[n]; elim: by the elimination alone.
__global__ void __launch_bounds__(32) solve_kernel(const double *sys, double pivot_eps, int elim, double *xi, int *ok) {
    __shared__ double tot[32];
    const int lane = threadIdx.x;
    tot[lane] = lane < 27 ? sys[(size_t)blockIdx.x * 27 + lane] : 0.0;
    __syncwarp();
    double x = 0.0;
    const bool r = elim ? warp_solve6_pivots(tot, pivot_eps, &x) : warp_solve6(tot, pivot_eps, &x);
    if (lane < 6) xi[(size_t)blockIdx.x * 6 + lane] = x;
    if (lane == 0) ok[blockIdx.x] = r ? 1 : 0;
}
}  // namespace upslam

extern "C" int probe_solve(const double *d_sys, int n, double pivot_eps, int elim, double *d_xi, int *d_ok) {
    upslam::solve_kernel<<<n, 32>>>(d_sys, pivot_eps, elim, d_xi, d_ok);
    return cudaDeviceSynchronize() == cudaSuccess ? 0 : 1;
}

// The kernels' binning of points given as such, and the plain rule's: tests/test_gpu_bin_pixel.py builds and loads it.
#include "../paper_2101_00585_gb300/csrc/common.cuh"

namespace upslam {
__global__ void __launch_bounds__(256) bin_kernel(const float4 *pts, int n, BinRule b, int *cell, int *rule) {
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        const float4 p = pts[i];
        cell[i] = bin_pixel(p.x, p.y, p.z, b);
        int row, col;
        float r;
        rule[i] = bin_point(p.x, p.y, p.z, b.pp, row, col, r) ? row * b.pp.cols + col : -1;
    }
}
}  // namespace upslam

extern "C" int probe_bin(const float *d_pts, int n, const upslam_pano *pp, int *d_cell, int *d_rule) {
    upslam::bin_kernel<<<1024, 256>>>(reinterpret_cast<const float4 *>(d_pts), n, make_bin_rule(*pp), d_cell, d_rule);
    return cudaDeviceSynchronize() == cudaSuccess ? 0 : 1;
}

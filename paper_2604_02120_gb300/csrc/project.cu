// Preprocessing stage (Sec. 2.1 (a)): EWA projection of 3D Gaussians, one
// thread per Gaussian.  FP32 throughout; the 2D covariance and its inverse are
// recomputed in FP64 when the FP32 determinant is below 1e-6.
#include <algorithm>

#include "project.cuh"

namespace gs {
namespace {

// Blocks run chunk by chunk of Gaussians (grid z), within a chunk view by view (y),
// so that a chunk's inputs come from HBM once and its other views read them from
// L2; outputs of view v, Gaussian g at index v * n + g.  How many blocks a chunk
// has is a matter of what moves.  Degrees 0 and 1 write nearly as much as they
// read, and every view's outputs are streams of their own: whole waves per view
// (1024 blocks, 131072 Gaussians).  Degree 3 is bound by the coefficients, which 16
// blocks keep closest; degree 2 lies between (16 views of 200k 98 us in chunks of 16,
// 94 in chunks of 1024; two views of 3M 204 and 209).  Degree 0, 16 views of 300k /
// 1.5M: view by view over all Gaussians 74 / 567 us, views innermost (chunks of one
// block) 107 / 514, in chunks of 1024 74 / 340; degree 3, 16 views of 1.5M: 1124, 747,
// 787, in chunks of 16 748 (5 views of 3M 710, 514, 524, 500).
// Bound by the latency of a chain of loads (means, then shape, then the
// coefficients of what is visible), so by resident warps: 64 registers and small
// blocks.  3M Gaussians, degree 3, one view 146 -> 127 us (663 MB, 5.2 TB/s).
constexpr int kProjThreads = 128;
constexpr unsigned chunk_blocks(int sh_degree, int views) {
    return sh_degree <= 1 || (sh_degree == 2 && views > 2) ? 1024 : 16;
}
template <int SH_DEGREE, bool VEC16>
__global__ void __launch_bounds__(kProjThreads, 8) k_project(int n, const float* __restrict__ means,
                                                 const float* __restrict__ scales, const float* __restrict__ quats,
                                                 const float* __restrict__ sh,
                                                 const __grid_constant__ CamViews views,
                                                 float2* __restrict__ mean2d_all, float* __restrict__ conic_all,
                                                 float* __restrict__ depth_all, int* __restrict__ radius_all,
                                                 float* __restrict__ rgb_all, uint32_t* __restrict__ touched_all) {
    const unsigned g = (blockIdx.z * gridDim.x + blockIdx.x) * kProjThreads + threadIdx.x, v = blockIdx.y;
    if (g >= (unsigned)n) return;
    project_gaussian<SH_DEGREE, VEC16>((int)g, means, scales, quats, sh, views.cams[v], (size_t)v * n,
                                       mean2d_all, conic_all, depth_all, radius_all, rgb_all, touched_all);
}

}  // namespace

cudaError_t launch_project(int n, const float* means, const float* scales, const float* quats, const float* sh,
                           int sh_degree, const CamViews& cams, float* mean2d, float* conic, float* depth,
                           int* radius, float* rgb, uint32_t* tiles_touched, cudaStream_t s) {
    const int block = kProjThreads;
    const unsigned nblk = ((unsigned)n + block - 1) / block;
    // (at most 65535 chunks; blocks split evenly, the last chunk may be a few short)
    const unsigned chunk = std::max(chunk_blocks(sh_degree, cams.num_views), (nblk + 65534) / 65535);
    const unsigned chunks = (nblk + chunk - 1) / chunk;
    const dim3 grid((nblk + chunks - 1) / chunks, cams.num_views, chunks);
    // 16-byte coefficient loads for degrees 1 and 3 (3K a multiple of 4) on an aligned array
    const bool vec = (reinterpret_cast<uintptr_t>(sh) & 15) == 0;
    switch (sh_degree) {
        case 0: k_project<0, false><<<grid, block, 0, s>>>(n, means, scales, quats, sh, cams, reinterpret_cast<float2*>(mean2d), conic, depth, radius, rgb,
                                       tiles_touched);
            break;
        case 1:
            if (vec) k_project<1, true><<<grid, block, 0, s>>>(n, means, scales, quats, sh, cams, reinterpret_cast<float2*>(mean2d), conic, depth, radius, rgb,
                                       tiles_touched);
            else k_project<1, false><<<grid, block, 0, s>>>(n, means, scales, quats, sh, cams, reinterpret_cast<float2*>(mean2d), conic, depth, radius, rgb,
                                       tiles_touched);
            break;
        case 2: k_project<2, false><<<grid, block, 0, s>>>(n, means, scales, quats, sh, cams, reinterpret_cast<float2*>(mean2d), conic, depth, radius, rgb,
                                       tiles_touched);
            break;
        default:
            if (vec) k_project<3, true><<<grid, block, 0, s>>>(n, means, scales, quats, sh, cams, reinterpret_cast<float2*>(mean2d), conic, depth, radius, rgb,
                                       tiles_touched);
            else k_project<3, false><<<grid, block, 0, s>>>(n, means, scales, quats, sh, cams, reinterpret_cast<float2*>(mean2d), conic, depth, radius, rgb,
                                       tiles_touched);
            break;
    }
    count_launches();
    return cudaGetLastError();
}

}  // namespace gs

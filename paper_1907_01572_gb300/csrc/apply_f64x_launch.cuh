// Per-degree launches of the FP64 apply on the tensor pipe.
#pragma once
#include "apply_f64x.cuh"

namespace dg {
namespace apply_detail {

// CTAs of a bucket's launch: as many as are resident at once, each taking elements in turn.
template <typename K>
LaunchShape x64_shape(K kernel, size_t smem) {
    LaunchShape r{};
    r.W = kX64Warps;
    r.smem = smem;
    r.err = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (r.err == cudaSuccess)
        r.err = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&r.per_sm, kernel, 32 * kX64Warps, smem);
    if (r.err == cudaSuccess && r.per_sm < 1) r.err = cudaErrorInvalidConfiguration;
    return r;
}

template <int N>
cudaError_t launch_x64_trace(const LevelView<double>& L, const BucketInfo& b, const double* x, cudaStream_t st) {
    static const LaunchShape shp = x64_shape(x64_trace_kernel<N>, X64Layout<N, kX64Warps>::TSIZE * sizeof(double));
    if (shp.err != cudaSuccess) return shp.err;
    const int grid = std::min(b.count, grid_cap() * shp.per_sm);
    x64_trace_kernel<N><<<grid, 32 * kX64Warps, shp.smem, st>>>(L, b.desc, b.count, x);
    return cudaGetLastError();
}

template <int N>
cudaError_t launch_x64_element(const LevelView<double>& L, const BucketInfo& b, const double* x, double* y,
                               cudaStream_t st) {
    static const LaunchShape shp = x64_shape(x64_element_kernel<N>, X64Layout<N, kX64Warps>::ESIZE * sizeof(double));
    if (shp.err != cudaSuccess) return shp.err;
    const int grid = std::min(b.count, grid_cap() * shp.per_sm);
    x64_element_kernel<N><<<grid, 32 * kX64Warps, shp.smem, st>>>(L, b.desc, b.count, x, y);
    return cudaGetLastError();
}

#define DG_X64_INSTANCE(N)                                                                                    \
    template cudaError_t launch_x64_trace<N>(const LevelView<double>&, const BucketInfo&, const double*,      \
                                             cudaStream_t);                                                   \
    template cudaError_t launch_x64_element<N>(const LevelView<double>&, const BucketInfo&, const double*,    \
                                               double*, cudaStream_t);

}  // namespace apply_detail
}  // namespace dg

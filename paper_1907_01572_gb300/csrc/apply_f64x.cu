// Launches of the FP64 apply on the tensor pipe (apply_f64x.cuh).
#include "apply_f64x.cuh"

namespace dg {
namespace apply_detail {

// All degree buckets in one launch (levels whose buckets alone leave SMs idle).
__global__ void __launch_bounds__(32 * kX64FusedWarps, 3) x64_trace_fused(LevelView<double> L, FusedBuckets fb, const double* __restrict__ x) {
    const int b = fused_bucket(fb);
    DG_BODY_SWITCH(fb.n[b], (x64_trace_body<NN, kX64FusedWarps>(L, fb.desc[b], fb.count[b], x, blockIdx.x - fb.cta_start[b],
                                                      fb.cta_start[b + 1] - fb.cta_start[b])))
}
__global__ void __launch_bounds__(32 * kX64FusedWarps, 3)
    x64_element_fused(LevelView<double> L, FusedBuckets fb, const double* __restrict__ x, double* __restrict__ y) {
    const int b = fused_bucket(fb);
    DG_BODY_SWITCH(fb.n[b], (x64_element_body<NN, kX64FusedWarps>(L, fb.desc[b], fb.count[b], x, y, blockIdx.x - fb.cta_start[b],
                                                        fb.cta_start[b + 1] - fb.cta_start[b])))
}

cudaError_t launch_x64_fused(const LevelView<double>& L, const BucketInfo* buckets, const double* x, double* y,
                             cudaStream_t st, int* launches) {
    size_t smem_t = 0, smem_e = 0;
    FusedBuckets fb{};
    int ctas = 0;
    for (int n = kMaxN; n >= kMinN; --n) {   // the longest elements first
        const BucketInfo& b = buckets[n];
        if (b.count == 0) continue;
        size_t t = 0, e = 0;
        DG_N_SWITCH(n, (t = X64Layout<NN, kX64FusedWarps>::TSIZE, e = X64Layout<NN, kX64FusedWarps>::ESIZE))
        smem_t = std::max(smem_t, t * sizeof(double));
        smem_e = std::max(smem_e, e * sizeof(double));
        fb.n[fb.nb] = n;
        fb.desc[fb.nb] = b.desc;
        fb.count[fb.nb] = b.count;
        fb.cta_start[fb.nb] = ctas;
        ctas += b.count;
        ++fb.nb;
    }
    fb.cta_start[fb.nb] = ctas;
    static const cudaError_t attr = [] {
        const int cap = 220 * 1024;
        const cudaError_t e1 = cudaFuncSetAttribute(x64_trace_fused, cudaFuncAttributeMaxDynamicSharedMemorySize, cap);
        const cudaError_t e2 = cudaFuncSetAttribute(x64_element_fused, cudaFuncAttributeMaxDynamicSharedMemorySize, cap);
        return e1 != cudaSuccess ? e1 : e2;
    }();
    if (attr != cudaSuccess) return attr;
    x64_trace_fused<<<ctas, 32 * kX64FusedWarps, smem_t, st>>>(L, fb, x);
    cudaError_t err = cudaGetLastError();
    if (err != cudaSuccess) return err;
    x64_element_fused<<<ctas, 32 * kX64FusedWarps, smem_e, st>>>(L, fb, x, y);
    if (launches) *launches += 2;
    return cudaGetLastError();
}

}  // namespace apply_detail

cudaError_t launch_apply_x64(const LevelView<double>& L, const BucketInfo* buckets, const double* x, double* y,
                             cudaStream_t st, int* launches, const ApplyStreams* as) {
    using namespace apply_detail;
    if (L.Ob != nullptr) {
        const cudaError_t err = launch_galerkin_apply<double, double>(L, buckets, x, y, st, launches);
        if (err != cudaSuccess) return err;
    }
    int degrees = 0;
    for (int n = kMinN; n <= kMaxN; ++n) degrees += buckets[n].count > 0;
    if (degrees > 1 && L.n_elems <= kX64FusedMaxElems) return launch_x64_fused(L, buckets, x, y, st, launches);
    return for_buckets(buckets, st, launches, as, [&](int phase, int n, cudaStream_t sj) {
        const BucketInfo& b = buckets[n];
        cudaError_t err = cudaSuccess;
        if (phase == 0) {
            DG_N_SWITCH(n, (err = launch_x64_trace<NN>(L, b, x, sj)))
        } else {
            DG_N_SWITCH(n, (err = launch_x64_element<NN>(L, b, x, y, sj)))
        }
        return err;
    });
}

}  // namespace dg

// Operator-apply launcher.
#pragma once
#include "internal.h"

namespace dg {

struct BucketInfo {        // elements of one degree on one level
    const int* elems;      // device element ids
    const ElemDesc* desc;  // device, per element of the bucket
    int count;
    int max_q;             // largest mortar q among the bucket's slots
    int max_nb;            // largest neighbour n among the bucket's slots
};

// Side streams on which per-degree bucket kernels run next to those on the
// caller's stream, so that one bucket's last elements overlap the next
// bucket's first (fork and join by events; capturable into CUDA graphs).
constexpr int kApplySide = 5;          // capacity (DGELL_APPLY_STREAMS=k, k <= 5, uses k)
constexpr int kApplySideDefault = 1;   // two-way overlap measured fastest on the 32^3 sweep mesh
struct ApplyStreams {
    int n = 0;                                   // side streams in use (0: the caller's stream only)
    cudaStream_t side[kApplySide] = {};
    cudaEvent_t fork[2] = {};                    // trace phase, element phase
    cudaEvent_t join[2][kApplySide] = {};
};
cudaError_t apply_streams_create(ApplyStreams& as);
void apply_streams_destroy(ApplyStreams& as);

// y = L x on one level; buckets indexed by n (2..9).  launches: incremented per kernel launch.
// plan: the level's launch-plan slot (-1 = not tuned yet; tuned on first use) or nullptr.
// as: side streams for the per-bucket launch plan, or nullptr.
template <typename T>
cudaError_t launch_apply(const LevelView<T>& L, const BucketInfo* buckets, const T* x, T* y, cudaStream_t st,
                         int* launches, int* plan = nullptr, const ApplyStreams* as = nullptr);

// Levels of at most this many elements (four per SM) hold the neighbours' records
// that the one-launch FP32 apply (apply_one.cuh) needs; whether it is the fastest
// on a level is measured with the other plans.  Alone it is faster beyond (1,056
// elements: 58 us against 65), but there the traces computed twice cost other
// streams their share: with three contexts in flight 832 elements took 41 us a
// pass against 33, 512 elements 15.0 against 15.7.
constexpr int kOneMaxElems = 608;

// FP64 with the contractions on the tensor pipe (apply_f64x.cuh): levels of at
// least kX64MinElems elements, two per SM, where the chip is full enough for the
// digits' throughput to count more than an element's latency.  Native against
// digits (us): 64 elements of p = 3 20 | 31, p = 5 35 | 56, p = 7 50 | 62; 120 hp
// elements 68 | 62; 160 of the level-1 cubed sphere 103 | 161; 512 elements of p = 3
// 64 | 41, p = 7 304 | 78.  (That sphere's V-cycle with the CG eigenvalue estimate
// amplifies rounding 1e8 times; below the line its FP64 results keep their bits.)
// Up to kX64FusedMaxElems elements the degrees share one launch (960 hp elements:
// 133 us against 299 in a launch per degree, 1,056 of the cubed sphere 303 against
// 508; 7,680: 723 against 562).
constexpr int kX64MinElems = 305;
constexpr int kX64FusedMaxElems = 2048;
// Low degrees stay native: a tile takes its time however little of it is used (a
// face of p = 1 fills 4 of 64 points), where the native kernels' work shrinks.  The
// line, native against digits (us): means of 17 DOFs per element (p 1..2) 66 | 86
// on 960 elements, 273 | 323 on 7,680, 1795 | 2353 on 61,440; 33 (p 1..3) 77 | 83,
// 330 | 338, 2209 | 2437; 45 (p 2..3) 80 | 80, 360 | 345; 56 (p 1..4) 385 | 354; 64 (p =
// 3) 224 | 174, 1449 | 1301.  Alone on a level and not too many, p = 1 and 2 are the
// exception: p = 1 42 | 40 at 512 elements, 129 | 157 at 4,096; p = 2 54 | 40, 175 |
// 164, and 1079 | 1242 at 32,768.
inline bool x64_pays(int n_elems, const BucketInfo* buckets) {
    if (n_elems < kX64MinElems) return false;
    long long dofs = 0;
    int degrees = 0, top = 0;
    for (int n = kMinN; n <= kMaxN; ++n) {
        if (buckets[n].count == 0) continue;
        dofs += (long long)buckets[n].count * n * n * n;
        ++degrees;
        top = n;
    }
    return dofs >= 40LL * n_elems || (degrees == 1 && n_elems <= (top == 2 ? 1024 : 4096));
}
cudaError_t launch_apply_x64(const LevelView<double>& L, const BucketInfo* buckets, const double* x, double* y,
                             cudaStream_t st, int* launches, const ApplyStreams* as);

// BF16 operand x (2-byte bfloat16 values), FP32 arithmetic and FP32 y.
cudaError_t launch_apply_bf16(const LevelView<float>& L, const BucketInfo* buckets, const void* x, float* y,
                              cudaStream_t st, int* launches, int* plan = nullptr,
                              const ApplyStreams* as = nullptr);

}  // namespace dg

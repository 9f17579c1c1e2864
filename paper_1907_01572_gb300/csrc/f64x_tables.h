// Digit tables of the FP64 apply on the tensor pipe (apply_f64x.cuh).
#pragma once
#include "internal.h"

namespace dg {

constexpr int kX64Digits = 6;

// Words of one operator (nc rows, k operands): per group of 8 rows and 8
// operands and digit, the half2 words of the 32 lanes of an mma.sync B fragment.
__host__ __device__ constexpr int x64_op_words(int nc, int k) {
    return ((nc + 7) / 8) * ((k + 7) / 8) * kX64Digits * 32;
}

// Volume operators of n: I, I^T, Dg, Dg^T and the two end rows of DL.
enum X64Vol { kX64I = 0, kX64IT, kX64D, kX64DT, kX64Ends, kX64NumVol };
__host__ __device__ constexpr int x64_vol_off(int n, int op) {
    int o = 0;
    for (int m = kMinN; m < n; ++m) o += kX64NumVol * x64_op_words(m, m);
    return o + op * x64_op_words(n, n);
}
// Mortar operators of a side n and mortar q >= n: op 0 Im, 1 Dm, 2 Im^T, 3 Dm^T, sub-face pos.
__host__ __device__ constexpr int x64_face_off(int n, int q, int pos, int op) {
    int o = x64_vol_off(kMaxN + 1, 0);
    for (int m = kMinN; m <= n; ++m)
        for (int r = m; r < (m < n ? kMaxN + 1 : q); ++r) o += 12 * x64_op_words(r, m);
    return o + (pos * 4 + op) * x64_op_words(q, n);
}
constexpr int kX64Words = x64_face_off(kMaxN, kMaxN, 2, 3) + x64_op_words(kMaxN, kMaxN);

// Scales (the tables hold R 2^-s): kX64NumVol per n, then 4 per (n, q).
__host__ __device__ constexpr int x64_vol_scale(int n) { return kX64NumVol * (n - kMinN); }
__host__ __device__ constexpr int x64_face_scale(int n, int q) {
    return kX64NumVol * kNumN + 4 * ((n - kMinN) * kNumN + (q - kMinN));
}
constexpr int kX64Scales = kX64NumVol * kNumN + 4 * kNumN * kNumN;

// From the 1-D tables (build_tables); false if a sum of digit products could
// leave the exact range of the accumulators.
bool build_x64_tables(const std::vector<double>& tab, std::vector<unsigned>& w, std::vector<int>& s);

}  // namespace dg

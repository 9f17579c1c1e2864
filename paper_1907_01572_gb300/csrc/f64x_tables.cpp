// Digit tables of the FP64 apply on the tensor pipe (f64x_tables.h).
#include <cuda_fp16.h>

#include <algorithm>
#include <cmath>

#include "f64x_tables.h"

namespace dg {
namespace {

// Digit pairs summed in one accumulator (apply_f64x.cuh, tile_product): the
// operator's digits j in each (level 6, scaled by 2^-10, adds less than
// 8192 to the first three).
const int kGroups[10][3] = {{5, 4, -1}, {3, 2, -1}, {1, 0, -1}, {4, 3, -1}, {2, 1, 0},
                            {3, 2, -1}, {1, 0, -1}, {2, 1, 0}, {1, 0, -1}, {0, -1, -1}};

int scale_of(const std::vector<std::vector<double>>& ops, int nc, int k) {
    double l1 = 0.0;
    for (const auto& R : ops)
        for (int i = 0; i < nc; ++i) {
            double s = 0.0;
            for (int j = 0; j < k; ++j) s += std::fabs(R[i * k + j]);
            l1 = std::max(l1, s);
        }
    int s = 0;
    while (std::ldexp(l1, -s) > 1.0) ++s;
    return s;
}

bool put(const std::vector<double>& R, int nc, int k, int s, unsigned* w) {
    std::vector<int> d((size_t)kX64Digits * nc * k);
    for (int i = 0; i < nc * k; ++i) {
        double x = std::ldexp(R[i], 9 - s);
        for (int j = 0; j < kX64Digits; ++j) {   // exact: each digit is the nearest integer to what is left
            const double v = std::nearbyint(x);
            d[(size_t)j * nc * k + i] = (int)v;
            x = (x - v) * 1024.0;
        }
    }
    for (const auto& grp : kGroups)
        for (int i = 0; i < nc; ++i) {
            long long sum = 0;
            for (int j : grp)
                for (int c = 0; j >= 0 && c < k; ++c) sum += std::abs(d[(size_t)j * nc * k + i * k + c]);
            if (512 * sum >= (1 << 22) - 8192) return false;
        }
    const int nt = (nc + 7) / 8, kg = (k + 7) / 8;
    for (int a = 0; a < nt; ++a)
        for (int b = 0; b < kg; ++b)
            for (int j = 0; j < kX64Digits; ++j)
                for (int lane = 0; lane < 32; ++lane) {
                    unsigned word = 0;
                    for (int h = 0; h < 2; ++h) {
                        const int row = 8 * a + (lane >> 2), col = 8 * b + 2 * (lane & 3) + h;
                        const int v = row < nc && col < k ? d[(size_t)j * nc * k + row * k + col] : 0;
                        __half_raw hr = __half_raw(__float2half((float)v));
                        word |= (unsigned)hr.x << (16 * h);
                    }
                    w[((a * kg + b) * kX64Digits + j) * 32 + lane] = word;
                }
    return true;
}

std::vector<double> transposed(const std::vector<double>& R, int nc, int k) {
    std::vector<double> t(R.size());
    for (int i = 0; i < nc; ++i)
        for (int j = 0; j < k; ++j) t[j * nc + i] = R[i * k + j];
    return t;
}

}  // namespace

bool build_x64_tables(const std::vector<double>& tab, std::vector<unsigned>& w, std::vector<int>& s) {
    w.assign(kX64Words, 0u);
    s.assign(kX64Scales, 0);
    bool ok = true;
    for (int n = kMinN; n <= kMaxN; ++n) {
        auto mat = [&](int base) {
            const double* p = &tab[tab_n(base, n)];
            return std::vector<double>(p, p + n * n);
        };
        const std::vector<double> I = mat(TabIndex::I), D = mat(TabIndex::Dg), L = mat(TabIndex::DL);
        std::vector<double> ends(L.begin(), L.begin() + n);
        ends.insert(ends.end(), L.end() - n, L.end());
        const std::vector<double> ops[kX64NumVol] = {I, transposed(I, n, n), D, transposed(D, n, n), ends};
        for (int op = 0; op < kX64NumVol; ++op) {
            const int nc = op == kX64Ends ? 2 : n, sc = scale_of({ops[op]}, nc, n);
            s[x64_vol_scale(n) + op] = sc;
            ok = put(ops[op], nc, n, sc, &w[x64_vol_off(n, op)]) && ok;
        }
        for (int q = n; q <= kMaxN; ++q) {
            std::vector<std::vector<double>> R[4];
            for (int pos = 0; pos < 3; ++pos)
                for (int t = 0; t < 2; ++t) {
                    const double* p = &tab[tab_m(t == 0 ? TabIndex::Im : TabIndex::Dm, n, q, pos)];
                    const std::vector<double> m(p, p + q * n);
                    R[t].push_back(m);
                    R[2 + t].push_back(transposed(m, q, n));
                }
            for (int op = 0; op < 4; ++op) {
                const int nc = op < 2 ? q : n, k = op < 2 ? n : q, sc = scale_of(R[op], nc, k);
                s[x64_face_scale(n, q) + op] = sc;
                for (int pos = 0; pos < 3; ++pos) ok = put(R[op][pos], nc, k, sc, &w[x64_face_off(n, q, pos, op)]) && ok;
            }
        }
    }
    return ok;
}

}  // namespace dg

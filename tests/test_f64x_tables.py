"""Digit tables of the FP64 apply on the tensor pipe (host code, no GPU): they
can be built for every degree and mortar size -- else the apply would fall back
to the FP64 kernels unnoticed -- and the digits add up to the operators."""
import os
import shutil
import subprocess

import pytest

from paper_1907_01572_gb300 import build

SOURCE = r"""
#include <cmath>
#include <cstdio>
#include <cuda_fp16.h>
#include "f64x_tables.h"
using namespace dg;
static double worst = 0.0;
static void check(const std::vector<unsigned>& w, int off, int scale, int nc, int k, const double* R, int r, int c) {
    for (int i = 0; i < nc; ++i)
        for (int j = 0; j < k; ++j) {
            double v = 0.0;   // digits from the smallest up: exact
            for (int d = kX64Digits - 1; d >= 0; --d) {
                const int a = i / 8, b = j / 8, lane = 4 * (i % 8) + (j % 8) / 2;
                const unsigned word = w[off + ((a * ((k + 7) / 8) + b) * kX64Digits + d) * 32 + lane];
                __half_raw h;
                h.x = (unsigned short)(word >> (16 * (j % 2)));
                const double digit = __half2float(__half(h));
                if (std::fabs(digit) > 512 || digit != std::nearbyint(digit)) worst = 1.0;
                v += std::ldexp(digit, -10 * d);
            }
            worst = std::max(worst, std::fabs(std::ldexp(v, -9) - std::ldexp(R[i * r + j * c], -scale)));
        }
}
int main() {
    std::vector<double> tab;
    std::vector<unsigned> w;
    std::vector<int> s;
    build_tables(tab);
    const bool ok = build_x64_tables(tab, w, s);
    for (int n = kMinN; n <= kMaxN; ++n) {
        const double *I = &tab[tab_n(TabIndex::I, n)], *D = &tab[tab_n(TabIndex::Dg, n)], *E = &tab[tab_n(TabIndex::DL, n)];
        const int* vs = &s[x64_vol_scale(n)];
        check(w, x64_vol_off(n, kX64I), vs[kX64I], n, n, I, n, 1);
        check(w, x64_vol_off(n, kX64IT), vs[kX64IT], n, n, I, 1, n);
        check(w, x64_vol_off(n, kX64D), vs[kX64D], n, n, D, n, 1);
        check(w, x64_vol_off(n, kX64DT), vs[kX64DT], n, n, D, 1, n);
        check(w, x64_vol_off(n, kX64Ends), vs[kX64Ends], 2, n, E, n * (n - 1), 1);
        for (int q = n; q <= kMaxN; ++q)
            for (int pos = 0; pos < 3; ++pos)
                for (int op = 0; op < 4; ++op) {
                    const double* M = &tab[tab_m(op % 2 ? TabIndex::Dm : TabIndex::Im, n, q, pos)];
                    const int sc = s[x64_face_scale(n, q) + op];
                    if (op < 2) check(w, x64_face_off(n, q, pos, op), sc, q, n, M, n, 1);
                    else check(w, x64_face_off(n, q, pos, op), sc, n, q, M, 1, n);
                }
    }
    std::printf("%d %.17g\n", (int)ok, worst);
}
"""


def test_digit_tables(tmp_path):
    nvcc = build._nvcc()
    if not (os.path.isabs(nvcc) or shutil.which(nvcc)):
        pytest.skip("no nvcc")
    src = tmp_path / "tables.cpp"
    src.write_text(SOURCE)
    cmd = [nvcc, "-x", "cu"] + build.ARCH + build.FLAGS + ["-I" + build.CSRC, str(src)]
    cmd += [os.path.join(build.CSRC, f) for f in ("host_tables.cpp", "f64x_tables.cpp")] + ["-o", str(tmp_path / "tables")]
    subprocess.run(cmd, check=True, capture_output=True)
    ok, worst = subprocess.run([str(tmp_path / "tables")], check=True, capture_output=True, text=True).stdout.split()
    assert ok == "1"
    # six digits of 10 bits: a unit of 2^-59, rounded to the nearest
    assert float(worst) <= 2.0 ** -60

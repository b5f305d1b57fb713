"""The limb arithmetic of FP64 links (csrc/fixed64.cuh), compiled for the host: the third row that
recon-12 links are rebuilt with keeps the limbs within the bounds that the hops rely on."""
import os
import subprocess

import pytest

from paper_1810_04201_gb300 import build

SOURCE = r"""
#include <cstdio>
#include <random>
#include "fixed64.cuh"
using namespace wd;
typedef long double T;

static T value(int h, int l) { return (T)h * 0x1p-30L + (T)fx_float(l) * 0x1p-62L; }

int main() {
    std::mt19937_64 rng(1);
    std::normal_distribution<double> gauss;
    const float top = 0x1p31f - 128.f;  // the largest float below 2^31
    double worst_limb = 0, worst_err = 0;
    for (int trial = 0; trial < 200000; ++trial) {
        double v[6][2];  // rows 0 and 1 of a unitary matrix, re and im
        for (auto &e : v) e[0] = gauss(rng), e[1] = gauss(rng);
        for (int row = 0; row < 2; ++row) {
            double *r = v[3 * row];
            if (row)
                for (int pass = 0; pass < 2; ++pass) {
                    double re = 0, im = 0;
                    for (int k = 0; k < 3; ++k) {
                        re += v[k][0] * v[3 + k][0] + v[k][1] * v[3 + k][1];
                        im += v[k][0] * v[3 + k][1] - v[k][1] * v[3 + k][0];
                    }
                    for (int k = 0; k < 3; ++k) {
                        v[3 + k][0] -= re * v[k][0] - im * v[k][1];
                        v[3 + k][1] -= re * v[k][1] + im * v[k][0];
                    }
                }
            double n = 0;
            for (int k = 0; k < 6; ++k) n += r[k] * r[k];
            for (int k = 0; k < 6; ++k) r[k] /= std::sqrt(n);
        }
        int4 u[9];
        for (int e = 0; e < 6; ++e) {
            const int2 re = fx_link(v[e][0]), im = fx_link(v[e][1]);
            u[e] = make_int4(re.x, re.y, im.x, im.y);
        }
        if (trial % 3) {  // low limbs at the end of their range, of random sign, or ...
            for (int e = 0; e < 6; ++e) {
                u[e].y = fx_bits(rng() & 1 ? top : -top);
                u[e].w = fx_bits(rng() & 1 ? top : -top);
            }
            if (trial % 3 == 2) {  // ... all adding up in the real part of entry 6
                auto sgn = [&](double x) { return fx_bits(x < 0 ? -top : top); };
                const int a = 1, b = 5, c = 2, d = 4;
                u[b].y = sgn(v[a][0]);  u[a].y = sgn(v[b][0]);  u[b].w = sgn(-v[a][1]); u[a].w = sgn(-v[b][1]);
                u[d].y = sgn(-v[c][0]); u[c].y = sgn(-v[d][0]); u[d].w = sgn(v[c][1]);  u[c].w = sgn(v[d][1]);
            }
        }
        fx_row2(u);
        for (int k = 0; k < 3; ++k) {
            const int i = (k + 1) % 3, j = (k + 2) % 3;
            auto re = [&](int e) { return value(u[e].x, u[e].y); };
            auto im = [&](int e) { return value(u[e].z, u[e].w); };
            const T xr = re(i) * re(3 + j) - im(i) * im(3 + j) - re(j) * re(3 + i) + im(j) * im(3 + i);
            const T xi = re(i) * im(3 + j) + im(i) * re(3 + j) - re(j) * im(3 + i) - im(j) * re(3 + i);
            const double er = (double)fabsl(re(6 + k) - xr), ei = (double)fabsl(im(6 + k) + xi);
            worst_err = std::max(worst_err, std::max(er, ei));
            worst_limb = std::max(worst_limb, (double)std::max(fabsf(fx_float(u[6 + k].y)), fabsf(fx_float(u[6 + k].w))));
        }
    }
    printf("%.17g %.17g\n", worst_limb, worst_err);
    return 0;
}
"""


def test_rebuilt_rows_stay_within_the_limbs(tmp_path):
    """|L| <= 2^31 + 2^10 (before the carry 4.7 x 2^31).  The entry's error is the FP32 rounding of two
    chains of four cross products, whose sums stay below 2^62 in units 2^-92 (2^-54 a step), of their
    difference and of L before the carry, below 2^34 (2^-53 each); the products of low limbs, 2^-62
    each, are below that."""
    src = tmp_path / "limbs.cu"
    src.write_text("#include <algorithm>\n" + SOURCE)
    exe = tmp_path / "limbs"
    subprocess.run([build.nvcc(), "-std=c++17", "-O2", *build.ARCH, "--expt-relaxed-constexpr", "-I", build.CSRC,
                    str(src), "-o", str(exe)], check=True, capture_output=True)
    limb, err = map(float, subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout.split())
    assert limb <= 2.0 ** 31 + 2.0 ** 10
    assert err <= 12 * 2.0 ** -54

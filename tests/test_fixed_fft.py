"""The FP64 form's block fixed-point transforms (csrc/qhfpe_fixed.cuh, compiled for the host) against extended
precision: a forward transform, a product with a real table and the inverse transform of rows of several
shapes, among them a single spike, values over many binary orders, full-scale and denormal-near rows."""
import os
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1706_09590_gb300", "csrc")

SOURCE = r"""
#include "qhfpe_fixed.cuh"
#include <cmath>
#include <complex>
#include <cstdio>
#include <random>
#include <vector>
using namespace qhfx;
typedef long double LD;
typedef std::complex<LD> CL;
static void pass16(I2 *X, int n) { for (int g = 0; g < n; g += 16) dft16<+1>(X + g); }
// forward error over the row's norm, then that of the product's inverse over (largest table value) * norm
template <int R0> static void run(int kind, std::mt19937_64 &rng, double *worst)
{
    const int NP = 16 * R0;
    const LD tau = 2 * std::acos(-1.0L);
    std::vector<I2> w(NP), X(NP);
    std::vector<CL> e(NP);
    for (int t = 0; t < NP; ++t) {
        e[t] = CL(std::cos(tau * t / NP), std::sin(tau * t / NP));
        w[t] = I2{std::llrint(e[t].real() * 0x1p62L), std::llrint(e[t].imag() * 0x1p62L)};
    }
    std::uniform_real_distribution<double> u(-1, 1);
    std::vector<double> re(NP), im(NP), D(NP);
    const int spike = rng() % NP;
    for (int l = 0; l < NP; ++l) {
        const double a = u(rng), b = u(rng), g = std::exp(-0.5 * std::pow((l - NP * 0.45) / (0.1 * NP), 2));
        re[l] = kind == 0 ? a : kind == 1 ? g * std::cos(0.7 * l) : kind == 2 ? (l == spike) * a : kind == 3 ? a * std::exp(30 * b)
              : kind == 4 ? 1.0 - 1e-16 * (l & 1) : kind == 5 ? a * 1e-280 : ((l & 1) ? -0.999999 : 0.999999);
        im[l] = kind == 1 ? g * std::sin(0.7 * l) : kind == 4 ? 1.0 : kind == 2 ? (l == spike) * b : kind == 5 ? b * 1e-280 : b;
        D[l] = u(rng) * 37.0;
    }
    int E = common_exponent<256>(std::vector<double>(256, 0.0).data(), std::vector<double>(256, 0.0).data());
    for (int l = 0; l < NP; ++l) E = std::max(E, std::max(exponent_of(re[l]), exponent_of(im[l])));
    constexpr int B = Scale<R0>::bits;
    for (int l = 0; l < NP; ++l) X[l] = I2{to_fixed<B>(re[l], E), to_fixed<B>(im[l], E)};
    for (int j = 0; j < 16; ++j) {
        I2 x[16];
        for (int t = 0; t < R0; ++t) x[t] = X[j + 16 * t];
        forward_butterfly<R0>(x, w.data(), j);
        for (int t = 0; t < R0; ++t) X[j + 16 * t] = x[t];
    }
    pass16(X.data(), NP);
    std::vector<CL> f(NP);
    LD n2 = 0, d2 = 0;
    for (int p = 0; p < NP; ++p) {
        const int k = p / 16 + R0 * (p % 16);
        for (int l = 0; l < NP; ++l) f[p] += CL(re[l], im[l]) * e[(long)k * l % NP];
        n2 += std::norm(f[p]);
        const int K = E + Scale<R0>::K_fwd + 2;
        d2 += std::norm(CL(from_fixed(X[p].x, K), from_fixed(X[p].y, K)) - f[p]);
    }
    worst[0] = std::max(worst[0], (double)std::sqrt(d2 / n2));
    // times the table (exponent k: values c 2^(k - 62)), parts exchanged, inverse
    double big = 0;
    for (double v : D) big = std::max(big, std::fabs(v));
    int k;
    std::frexp(big, &k);
    std::vector<int> er(16);
    for (int g = 0; g < R0; ++g) {  // a run of 16 modes
        unsigned o = 0, q = 0;
        for (int t = 0; t < 16; ++t) o |= magnitude(X[16 * g + t]);
        const int n = norm_shift<61>(o);
        for (int t = 0; t < 16; ++t) {
            const long long c = std::llrint(std::ldexp(D[16 * g + t], 62 - k));
            const I2 x = shift(X[16 * g + t], n);
            X[16 * g + t] = I2{mul_hi(x.y, c), mul_hi(x.x, c)};
            q |= magnitude(X[16 * g + t]);
        }
        const int m = norm_shift<59>(q);
        for (int t = 0; t < 16; ++t) X[16 * g + t] = shift(X[16 * g + t], m);
        er[g] = E - n + k - m;
    }
    pass16(X.data(), NP);
    std::vector<CL> y(NP);
    for (int j = 0; j < 16; ++j) {
        I2 x[16];
        for (int t = 0; t < R0; ++t) x[t] = X[j + 16 * t];
        const int K = align<R0>(x, er.data()) + Scale<R0>::K_fwd + 4 + 2 + Scale<R0>::inv + Scale<R0>::down;
        inverse_butterfly<R0>(x, w.data(), j);
        for (int t = 0; t < R0; ++t) y[j + 16 * t] = CL(from_fixed(x[t].y, K), from_fixed(x[t].x, K));
    }
    d2 = 0;
    for (int l = 0; l < NP; ++l) {
        CL a = 0;
        for (int p = 0; p < NP; ++p) a += f[p] * (LD)D[p] * std::conj(e[(long)(p / 16 + R0 * (p % 16)) * l % NP]);
        d2 += std::norm(y[l] - a);
    }
    worst[1] = std::max(worst[1], (double)(std::sqrt(d2 / (n2 * NP)) / big));
}
int main()
{
    std::mt19937_64 rng(1706);
    for (int kind = 0; kind < 7; ++kind) {
        double w[2] = {0, 0};
        for (int t = 0; t < 6; ++t) {
            run<2>(kind, rng, w);
            run<4>(kind, rng, w);
            run<8>(kind, rng, w);
            run<16>(kind, rng, w);
        }
        std::printf("%d %.3e %.3e\n", kind, w[0], w[1]);
    }
    // conversions: exact where 53 bits hold the value, and signs, zeros
    int bad = 0;
    for (double v : {0.0, 1.0, -1.0, 0.1, -7.25, 1e300, -3e-290, 4503599627370497.0}) {
        const int E = std::max(exponent_of(v), EXP_MIN);
        bad += from_fixed(to_fixed<60>(v, E), E - 1022 - 60) != v;
    }
    bad += to_fixed<60>(3e-310, EXP_MIN) != 0;
    std::printf("bad %d\n", bad);
}
"""

# a butterfly's integers carry at least 2^-55 of the row's largest input, a sum of 16 independent roundings of
# them 2^-53, and the result is rounded to 53 bits (1.1e-16): 1.5 eps forward; the product and the inverse
# add the same again.  FP64 butterflies: 1.1e-16 to 2.9e-16 forward on these rows.
FORWARD, BOTH = 3.4e-16, 6.8e-16


def test_fixed_point_transforms(tmp_path):
    src = tmp_path / "fixed.cpp"
    src.write_text(SOURCE)
    exe = tmp_path / "fixed"
    subprocess.run(["g++", "-O2", "-std=c++17", "-Wno-unknown-pragmas", "-I", CSRC, "-o", str(exe), str(src)], check=True)
    lines = subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout.split("\n")
    for line in lines[:7]:
        kind, fwd, both = line.split()
        assert float(fwd) < FORWARD, line
        assert float(both) < BOTH, line
    assert lines[7] == "bad 0"

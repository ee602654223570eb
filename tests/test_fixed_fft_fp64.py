"""The block fixed-point transforms of the FP64 form (csrc/qhfpe_fixed.cuh, compiled for the host) beside transforms of
the same radices in FP64, on the same rows: errors against extended precision, forward and over a round trip."""
import os
import subprocess

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
typedef std::complex<double> CD;

// length R by length-2 and length-4 steps, sign +, in doubles
static CD unit(int k, int n)
{
    const LD a = 2 * std::acos(-1.0L) * k / n;
    return CD((double)std::cos(a), (double)std::sin(a));
}
template <int R> static void dft(CD *x)
{
    if constexpr (R == 2) {
        const CD t = x[0];
        x[0] = t + x[1];
        x[1] = t - x[1];
    } else if constexpr (R == 4) {
        const CD a = x[0] + x[2], b = x[0] - x[2], c = x[1] + x[3], d = x[1] - x[3], id(-d.imag(), d.real());
        x[0] = a + c;
        x[2] = a - c;
        x[1] = b + id;
        x[3] = b - id;
    } else {  // R = 4 * Q
        constexpr int Q = R / 4;
        CD y[4][Q];
        for (int q = 0; q < Q; ++q) {
            CD t[4] = {x[q], x[q + Q], x[q + 2 * Q], x[q + 3 * Q]};
            dft<4>(t);
            for (int k = 0; k < 4; ++k) y[k][q] = q * k ? t[k] * unit(q * k, R) : t[k];
        }
        for (int k = 0; k < 4; ++k) {
            dft<Q>(y[k]);
            for (int l = 0; l < Q; ++l) x[k + 4 * l] = y[k][l];
        }
    }
}

template <int R0> struct Run {
    static constexpr int NP = 16 * R0;
    std::vector<CL> e;
    std::vector<I2> w;
    Run() : e(NP), w(NP)
    {
        for (int t = 0; t < NP; ++t) {
            const LD a = 2 * std::acos(-1.0L) * t / NP;
            e[t] = CL(std::cos(a), std::sin(a));
            w[t] = I2{std::llrint(e[t].real() * 0x1p62L), std::llrint(e[t].imag() * 0x1p62L)};
        }
    }
    static int frequency(int p) { return p / 16 + R0 * (p % 16); }
    void fp64(std::vector<CD> &x) const  // forward, digit-reversed order
    {
        for (int j = 0; j < 16; ++j) {
            CD t[R0];
            for (int u = 0; u < R0; ++u) t[u] = x[j + 16 * u];
            dft<R0>(t);
            for (int u = 0; u < R0; ++u)
                x[j + 16 * u] = u * j ? t[u] * CD((double)e[u * j].real(), (double)e[u * j].imag()) : t[u];
        }
        for (int g = 0; g < NP; g += 16) dft<16>(x.data() + g);
    }
    void fp64_back(std::vector<CD> &x) const  // and back, times NP (of exchanged parts, a forward one)
    {
        for (int g = 0; g < NP; g += 16) dft<16>(x.data() + g);
        for (int j = 0; j < 16; ++j) {
            CD t[R0];
            for (int u = 0; u < R0; ++u)
                t[u] = u * j ? x[j + 16 * u] * CD((double)e[u * j].real(), (double)e[u * j].imag()) : x[j + 16 * u];
            dft<R0>(t);
            for (int u = 0; u < R0; ++u) x[j + 16 * u] = t[u];
        }
    }
    void row(int kind, std::mt19937_64 &rng, double *s) const  // summed squared errors: fixed, FP64 forward; fixed, FP64 both ways
    {
        std::uniform_real_distribution<double> u(-1, 1);
        std::vector<CD> x(NP);
        const int spike = rng() % NP;
        for (int l = 0; l < NP; ++l) {
            const double a = u(rng), b = u(rng), g = std::exp(-0.5 * std::pow((l - NP * 0.45) / (0.1 * NP), 2));
            x[l] = kind == 0 ? CD(a, b) : kind == 1 ? CD(g * std::cos(0.7 * l), g * std::sin(0.7 * l))
                 : kind == 2 ? (l == spike ? CD(a, b) : CD()) : kind == 3 ? CD(a * std::exp(30 * b), b) : CD((l & 1) ? -a : a, 0.0);
        }
        std::vector<CL> f(NP);
        LD n2 = 0, in2 = 0;
        for (int p = 0; p < NP; ++p) {
            for (int l = 0; l < NP; ++l) f[p] += CL(x[l].real(), x[l].imag()) * e[(long)frequency(p) * l % NP];
            n2 += std::norm(f[p]);
            in2 += std::norm(CL(x[p].real(), x[p].imag()));
        }
        // fixed point
        int E = EXP_MIN;
        for (CD v : x) E = std::max(E, std::max(exponent_of(v.real()), exponent_of(v.imag())));
        constexpr int B = Scale<R0>::bits;
        std::vector<I2> X(NP);
        for (int l = 0; l < NP; ++l) X[l] = I2{to_fixed<B>(x[l].real(), E), to_fixed<B>(x[l].imag(), E)};
        for (int j = 0; j < 16; ++j) {
            I2 t[R0];
            for (int q = 0; q < R0; ++q) t[q] = X[j + 16 * q];
            forward_butterfly<R0>(t, w.data(), j);
            for (int q = 0; q < R0; ++q) X[j + 16 * q] = t[q];
        }
        for (int g = 0; g < NP; g += 16) dft16<+1>(X.data() + g);
        LD d = 0;
        const int K = E + Scale<R0>::K_fwd + 2;
        for (int p = 0; p < NP; ++p) d += std::norm(CL(from_fixed(X[p].x, K), from_fixed(X[p].y, K)) - f[p]);
        s[0] += (double)(d / n2);
        std::vector<int> er(R0);
        for (int g = 0; g < R0; ++g) {
            unsigned o = 0;
            for (int t = 0; t < 16; ++t) o |= magnitude(X[16 * g + t]);
            const int n = norm_shift<59>(o);
            for (int t = 0; t < 16; ++t) {
                const I2 v = shift(X[16 * g + t], n);
                X[16 * g + t] = I2{v.y, v.x};
            }
            er[g] = E - n;
        }
        for (int g = 0; g < NP; g += 16) dft16<+1>(X.data() + g);
        d = 0;
        for (int j = 0; j < 16; ++j) {
            I2 t[R0];
            for (int q = 0; q < R0; ++q) t[q] = X[j + 16 * q];
            const int Kb = align<R0>(t, er.data()) + Scale<R0>::K_fwd + 2 + 2 + Scale<R0>::inv + Scale<R0>::down;
            inverse_butterfly<R0>(t, w.data(), j);
            for (int q = 0; q < R0; ++q)
                d += std::norm(CL(from_fixed(t[q].y, Kb), from_fixed(t[q].x, Kb)) / (LD)NP -
                               CL(x[j + 16 * q].real(), x[j + 16 * q].imag()));
        }
        s[2] += (double)(d / in2);
        // doubles
        std::vector<CD> y = x;
        fp64(y);
        d = 0;
        for (int p = 0; p < NP; ++p) d += std::norm(CL(y[p].real(), y[p].imag()) - f[p]);
        s[1] += (double)(d / n2);
        for (CD &v : y) v = CD(v.imag(), v.real());
        fp64_back(y);
        d = 0;
        for (int l = 0; l < NP; ++l)
            d += std::norm(CL(y[l].imag(), y[l].real()) / (LD)NP - CL(x[l].real(), x[l].imag()));
        s[3] += (double)(d / in2);
    }
};
template <int R0> static void all(std::mt19937_64 &rng)
{
    const Run<R0> r;
    for (int kind = 0; kind < 5; ++kind) {
        double s[4] = {0, 0, 0, 0};
        for (int n = 0; n < 40; ++n) r.row(kind, rng, s);
        std::printf("%d %d", 16 * R0, kind);
        for (double v : s) std::printf(" %.3e", std::sqrt(v / 40));
        std::printf("\n");
    }
}
int main()
{
    std::mt19937_64 rng(42);
    all<2>(rng);
    all<4>(rng);
    all<8>(rng);
    all<16>(rng);
}
"""

# Root mean square over 40 rows.  The fixed-point transform's own rounding is below 2^-55 of the row's largest value a
# butterfly, its results are rounded to doubles once (at most 2^-53, 0.5 to 0.6 of that in the mean): no more than doubles' own
# representation error, while the FP64 butterflies round at every pass.  A spike (kind 2) is exact in FP64 but for the twiddle
# products.
REPRESENTATION = 2.0 ** -53


def test_fixed_point_against_fp64_butterflies(tmp_path):
    src = tmp_path / "fixed.cpp"
    src.write_text(SOURCE)
    exe = tmp_path / "fixed"
    subprocess.run(["g++", "-O2", "-std=c++17", "-Wno-unknown-pragmas", "-I", CSRC, "-o", str(exe), str(src)], check=True)
    out = subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout.strip().split("\n")
    assert len(out) == 20
    for line in out:
        n, kind, fixed, fp64, fixed2, fp64_2 = line.split()
        assert float(fixed) <= max(float(fp64), REPRESENTATION), line
        assert float(fixed2) <= max(float(fp64_2), REPRESENTATION), line

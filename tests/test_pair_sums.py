"""The FP32 sums that stand in for FP64 ones (csrc/ept_internal.cuh), compiled for the host from the
same header and checked against 64-bit and longer arithmetic."""
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def _program(d, name, body):
    """Compiles a main() that includes the header; no contraction, as the header's own rounding is under test."""
    src = d / (name + ".cu")
    src.write_text("#include <cmath>\n#include <cstdio>\n#include <cstdlib>\n#include <random>\n#include <vector>\n"
                   '#include "ept_internal.cuh"\n' + body)
    exe = d / name
    inc = os.path.join(ROOT, "paper_2406_06488_gb300", "csrc")
    try:
        subprocess.run([os.environ.get("NVCC", "nvcc"), "-O2", "-std=c++17", "-Xcompiler", "-ffp-contract=off",
                        "-I" + inc, "-o", str(exe), str(src)], check=True, capture_output=True)
    except OSError as e:
        pytest.skip("nvcc not usable here: %s" % e)
    return lambda *a: subprocess.run([str(exe)] + [str(x) for x in a], check=True, capture_output=True, text=True).stdout


# Two close rows of n features a pair: a root that SquareSum calls certain is the correctly rounded one (the sum lies
# between the squares of the midpoints to its neighbours), and few are left open.
ROOTS = r"""
int main(int argc, char **argv) {
    const int n = atoi(argv[1]), pairs = atoi(argv[2]);
    std::mt19937_64 g(n);
    std::normal_distribution<float> nd;
    long open = 0, wrong = 0;
    double worst = 0.0;   // the pair's error in units of its bound
    for (int q = 0; q < pairs; ++q) {
        ept::SquareSum s;
        long double S = 0;
        for (int k = 0; k < n; ++k) {
            const float base = 20.f * nd(g), x = base + nd(g), y = base + nd(g);
            s.add(x, y);
            if (k % 8 == 7) s.renormalise();
            const long double d = (long double)x - (long double)y;
            S += d * d;
        }
        s.renormalise();
        worst = std::fmax(worst, (double)(fabsl((long double)s.h + s.l - S) / S) / std::ldexp(41.0 * n, -48));
        float y;
        if (!s.root(n, y)) { ++open; continue; }
        const long double a = ((long double)y + nextafterf(y, 0.f)) / 2, b = ((long double)y + nextafterf(y, 1e30f)) / 2;
        wrong += !(a * a <= S && S <= b * b);
    }
    printf("%ld %ld %.17g\n", open, wrong, worst);
}
"""


@pytest.mark.parametrize("n,pairs", [(1, 40000), (3, 40000), (10, 40000), (257, 4000), (1500, 1000), (20000, 100)])
def test_certain_roots_are_rounded_right(tmp_path, n, pairs):
    left, wrong, worst = _program(tmp_path, "roots", ROOTS)(n, pairs).split()
    assert int(wrong) == 0 and float(worst) <= 1.0
    if n == 1:
        return   # one difference of 25 bits is the middle between two results itself
    # twice the bound over the spacing of the results (2^-23 to 2^-24 of them), and chance
    share = 2 * (21 * n + 32) * 2.0 ** -48 / 2.0 ** -24
    assert int(left) <= pairs * share + 5 * (pairs * share) ** 0.5 + 3


# Squared norms of rows of p features by L lanes, 4 elements a lane and step: a sum that NormSum calls certain is
# the correctly rounded one, and few are left open.  Last number: rows whose pair alone rounds the other way.
NORMS = r"""
int main(int argc, char **argv) {
    const int p = atoi(argv[1]), L = atoi(argv[2]), rows = atoi(argv[3]);
    std::mt19937_64 g(p + L);
    std::normal_distribution<float> nd;
    long open = 0, wrong = 0, plain = 0;
    double worst = 0.0;
    std::vector<float> z(p);
    for (int q = 0; q < rows; ++q) {
        long double S = 0;
        for (float &v : z) { v = nd(g); S += (long double)v * v; }
        std::vector<ept::NormSum> lane(L);
        for (int k = 0; k < p; ++k) lane[(k / 4) % L].add(z[k]);
        for (int off = L / 2; off; off /= 2)
            for (int k = 0; k < off; ++k) lane[k].merge(lane[k + off].h, lane[k + off].l);
        const float m6 = (float)(p / L + 10), want = (float)S;
        worst = std::fmax(worst, (double)(fabsl((long double)lane[0].h + lane[0].l - S) / S) / std::ldexp(2.0 * m6 * m6, -48));
        float y;
        plain += lane[0].h + lane[0].l != want;
        if (!lane[0].rounded(m6, y)) ++open;
        else wrong += y != want;
    }
    printf("%ld %ld %.17g %ld\n", open, wrong, worst, plain);
}
"""


@pytest.mark.parametrize("p,L,rows", [(1, 32, 40000), (5, 8, 40000), (100, 8, 40000), (512, 8, 20000), (1000, 32, 10000),
                                      (9001, 32, 1000), (200000, 32, 40)])
def test_certain_norms_are_rounded_right(tmp_path, p, L, rows):
    left, wrong, worst, _ = _program(tmp_path, "norms", NORMS)(p, L, rows).split()
    assert int(wrong) == 0 and float(worst) <= 1.0
    share = min(1.0, 8 * (p // L + 10) ** 2 * 2.0 ** -48 / 2.0 ** -24)
    assert int(left) <= rows * share + 5 * (rows * share) ** 0.5 + 3


# Sums of m partials over 2^20 in magnitude, of both signs or their magnitudes, exact in integers: the error within the bound and, in
# all, no larger than that of FP64 additions one by one.
TRIPLES = r"""
int main(int argc, char **argv) {
    const int m = atoi(argv[1]), sums = atoi(argv[2]);
    const bool magnitudes = atoi(argv[3]);
    std::mt19937_64 g(m);
    double worst = 0.0;
    long double err3 = 0, err64 = 0;
    for (int q = 0; q < sums; ++q) {
        ept::TripleSum s;
        double d = 0.0;
        long long S = 0, A = 0;
        for (int k = 0; k < m; ++k) {
            const long long v = (long long)(g() % (1 << 24)) << (g() % 21);
            const bool neg = (g() & 1) && !magnitudes;
            S += neg ? -v : v;
            A += v;
            s.add((float)(neg ? -v : v) * 0x1p-44f);
            d += (double)(neg ? -v : v) * 0x1p-44;
        }
        const long double want = (long double)S * 0x1p-44L, e = fabsl((long double)s.value() - want);
        err3 += e;
        err64 += fabsl((long double)d - want);
        const double bound = (double)m * m * m * 0x1p-72 * ((double)A * 0x1p-44) + 0x1p-52 * std::fabs((double)want);
        worst = std::fmax(worst, bound > 0 ? (double)e / bound : (double)e);
    }
    printf("%.17g %.17g %.17g\n", worst, (double)err3, (double)err64);
}
"""


@pytest.mark.parametrize("m", [1, 2, 7, 8, 9, 63, 64])
def test_triple_sums_lose_no_more_than_fp64(tmp_path, m):
    run = _program(tmp_path, "triples", TRIPLES)
    for magnitudes in (0, 1):
        worst, err3, err64 = (float(x) for x in run(m, 200000, magnitudes).split())
        assert worst <= 1.0 and err3 <= err64

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

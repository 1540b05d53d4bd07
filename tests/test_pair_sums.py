"""Float-pair arithmetic of the kernels (csrc/arith.h), compiled for the host:
errors against the same sums in extended precision."""
import os
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1712_02533_gb300", "csrc")

AVERAGE = r"""
#include <cmath>
#include <cstdio>
#include <random>
#include "arith.h"
// 3000 nodes averaged over m frames as the averaging kernel does it: the largest error
// over the stated tolerance, and the nodes whose rounding stays open (those are summed
// again in double).
int main()
{
    const int m = M, mode = MODE, nodes = 3000;
    std::mt19937 g(7);
    std::normal_distribution<double> z(0, 1);
    std::uniform_real_distribution<double> u(0.5, 4);
    double worst = 0;
    int open = 0;
    for (int t = 0; t < nodes; t++) {
        const double base = u(g), s0 = 5 + 3 * u(g), mean = 10 * u(g);
        PairSum s;
        long double exact = 0;
        double means = 0;
        for (int k = 0; k < m; k++) {
            // one sign and frames that differ; the same value in every frame; both signs
            const float v = (float)(mode == 0 ? base + 0.1 * z(g) : mode == 1 ? base : (k & 1 ? base : -base) + 1e-3 * z(g));
            const double sigma = mode == 1 ? s0 : s0 + 0.05 * z(g);
            const float sh = (float)sigma;
            s.add(v, sh, (float)(sigma - (double)sh));
            if ((k & 1) || k == m - 1) s.fold();
            exact += (long double)v * sigma;
            means += mean;
        }
        const double inv = 1.0 / m;
        const float ch = (float)means, cl = (float)(means - (double)ch), fh = (float)inv, fl = (float)(inv - (double)fh);
        float p, pl;
        s.scaled(ch, cl, fh, fl, p, pl);
        const float tol = s.tolerance(m, ch, fh);
        worst = std::fmax(worst, (double)std::fabs((long double)p + pl - (exact + means) / m) / tol);
        open += !(p + (pl - tol) == p + (pl + tol));
    }
    printf("%.9f %d\n", worst, open);
}
"""

ROOT = r"""
#include <cmath>
#include <cstdio>
#include <random>
#include "arith.h"
// 1 / sqrt, sqrt and S / sqrt of v over v's range, from seeds 2 ulp to either side of
// the float value: largest and root mean square relative errors in 2^-53, of the steps
// and of the square root and divisions of double precision.
int main()
{
    std::mt19937_64 g(3);
    std::uniform_real_distribution<double> u(0, 1);
    double mx[6] = {0}, ms[6] = {0};
    const int N = 2000000;
    for (int t = 0; t < N; t++) {
        // half of them around 1, where the variance of normalised frames lies
        const double v = t % 2 ? 0.25 + 2 * u(g) : std::exp2(-99 + 198 * u(g)), S = (2 * u(g) - 1) * std::sqrt(v);
        float r0 = (float)(1 / std::sqrt((long double)v));
        for (int k = t % 5 - 2; k != 0; k += k > 0 ? -1 : 1) r0 = std::nextafterf(r0, k > 0 ? INFINITY : 0.f);
        const long double s = std::sqrt((long double)v);
        const RootInv r = rsqrt_step(v, r0);
        const double q = std::sqrt(v);
        const long double got[6] = {r.r, times(v, r), times(S, r), 1 / q, q, S / q}, want[3] = {1 / s, s, S / s};
        for (int i = 0; i < 6; i++) {
            const double e = (double)std::fabs((got[i] - want[i % 3]) / want[i % 3]) * 9007199254740992.0;
            mx[i] = std::fmax(mx[i], e);
            ms[i] += e * e / N;
        }
    }
    for (int i = 0; i < 6; i++) printf("%.6f %.6f\n", mx[i], std::sqrt(ms[i]));
}
"""


def _run(tmp_path, src):
    (tmp_path / "t.cpp").write_text(src)
    subprocess.run(["g++", "-std=c++17", "-O2", "-ffp-contract=off", "-I", CSRC, str(tmp_path / "t.cpp"), "-o",
                    str(tmp_path / "t")], check=True)
    return subprocess.run([str(tmp_path / "t")], check=True, capture_output=True, text=True).stdout.split()


@pytest.mark.parametrize("mode", [0, 1, 2])
@pytest.mark.parametrize("m", [1, 2, 3, 64, 400, 4000])
def test_average_of_any_number_of_frames_keeps_its_tolerance(tmp_path, m, mode):
    """The error of the pair sum is at most the tolerance that decides whether a node's
    rounding is settled (derived beside the code; it grows with the number of frames m),
    and the open nodes stay few: a node is open with probability 2 (m + 4) 2^-45 / 2^-24
    times at most 4 (the result may be that much smaller than the terms' sum), 2% at
    4000 frames."""
    worst, n_open = _run(tmp_path, AVERAGE.replace("M,", f"{m},").replace("MODE,", f"{mode},"))
    assert float(worst) <= 1.0
    assert int(n_open) <= 0.05 * 3000


def test_reciprocal_root_is_as_accurate_as_root_and_division(tmp_path):
    """Over variances of 2^-99 to 2^99 and seeds as far off as rsqrtf may be: the
    reciprocal root is within 2^-53 (1 + 2^-10: what the third-order step leaves is
    below 2^-63), the root too, and neither they nor the quotient S / sqrt(v) are less
    accurate than square root and division of double precision, in the largest and
    in the mean error."""
    out = [float(x) for x in _run(tmp_path, ROOT)]
    step, plain = [out[2 * i:2 * i + 2] for i in range(3)], [out[2 * i + 6:2 * i + 8] for i in range(3)]
    assert step[0][0] <= 1 + 2.0 ** -10 and step[1][0] <= 1 + 2.0 ** -10
    for (mx, rms), (mx0, rms0) in zip(step, plain):
        # the largest of two million draws: to 1% of the bound of either form
        assert mx <= mx0 + 0.02 and rms <= 1.001 * rms0

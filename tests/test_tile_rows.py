"""Row ranges of the gradient pass's tiles (csrc/tile_rows.h), compiled for the
host: no warp loads a row outside its level, and every row has one owner."""
import os
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1712_02533_gb300", "csrc")

WALK = r"""
#include <cstdio>
#include <vector>
#include "tile_rows.h"
// The kernel's walk over every tile and warp: rows loaded off the level, rows whose
// neighbours were not loaded before they are completed, rows without exactly one owner.
int main()
{
    int off = 0, missing = 0, owners = 0;
    for (int l = 2; l <= 12; l++)
        for (int h : {4, 8, 16, 32, 64})
            for (int parts : {1, 4}) {
                const int n = (1 << l) + 1;
                std::vector<int> own(n, 0);
                for (int tile0 = 0; tile0 < n; tile0 += h)
                    for (int w = 0; w < parts; w++) {
                        const GradRows g = grad_rows(tile0, h, n, w, parts);
                        std::vector<char> got(n, 0);
                        auto load = [&](int r) {
                            if (r < 0 || r >= n) off++;
                            else got[r] = 1;
                        };
                        if (grad_loads_first(g.r0, n)) load(g.r0 - 1);
                        for (int r = g.r0 - 1; r <= g.rLast + 1; r++) {
                            if (r + 1 < n && r + 1 <= g.rLast + 1) load(r + 1);
                            const int m = r - 1;  // completed by row r
                            if (m < g.r0) continue;
                            if (m >= n) { owners++; continue; }
                            own[m]++;
                            for (int q = m - 1; q <= m + 1; q++)
                                if (q >= 0 && q < n && !got[q]) missing++;
                        }
                    }
                for (int r = 0; r < n; r++) owners += own[r] != 1;
            }
    printf("%d %d %d\n", off, missing, owners);
}
"""


@pytest.fixture(scope="module")
def compile_host(tmp_path_factory):
    def run(src):
        d = tmp_path_factory.mktemp("host")
        (d / "t.cpp").write_text(src)
        subprocess.run(["g++", "-std=c++17", "-O2", "-ffp-contract=off", "-I", CSRC, str(d / "t.cpp"), "-o", str(d / "t")],
                       check=True)
        return subprocess.run([str(d / "t")], check=True, capture_output=True, text=True).stdout.split()

    return run


def test_gradient_walks_stay_on_their_level(compile_host):
    """All levels of 2^2 + 1 to 2^12 + 1 rows, all tile heights, a tile per warp and
    a tile shared by four: no load off the level, every completed row with its
    neighbours at hand, every row completed by exactly one warp."""
    assert compile_host(WALK) == ["0", "0", "0"]


def test_a_batch_is_judged_by_its_widest_level(compile_host):
    """The most gradient tiles of an operator: on the finest level under the default
    rows (33 and 65 rows of 8, 129 and 257 of 16, 513 of 32), on the next one where the
    finest has 64 rows and that one 4."""
    src = """
#include <cstdio>
#include "tile_rows.h"
int main()
{
    const int n[5] = {33, 65, 129, 257, 513}, rows[5] = {8, 8, 16, 16, 32}, other[5] = {8, 8, 16, 4, 64};
    printf("%d %d %d\\n", most_grad_tiles(n, rows, 5, 30), most_grad_tiles(n, other, 5, 30), most_grad_tiles(n + 4, other + 4, 1, 30));
}
"""
    assert compile_host(src) == [str(18 * 17), str(9 * 65), str(18 * 9)]

"""The work plan of the pair-symmetric passes (csrc/pp_sym_plan.h, host code), checked by a
small C++ program: every source of every row is covered once, and no item of work is longer
than half a warp's share of what is left when it is handed out, whatever PP_OPT_SPLIT says
(the warps of a pass wait, bounded, for its last item)."""
import os
import shutil
import subprocess

import pytest

from paper_2502_10640_gb300 import build

DRIVER = r"""
#include <cstdio>
#include <cstdlib>
#include <functional>
#include <queue>
#include "pp_sym_plan.h"
using namespace ppk;
// argv: (n, targets, f64, slots, split)...; prints per plan: items, covered, over, longest,
// and the time until the last item ends over the even share of the work, items handed out in
// order to warps of one speed
int main(int argc, char **argv)
{
    for (int a = 1; a + 4 < argc; a += 5) {
        const int n = atoi(argv[a]), targets = atoi(argv[a + 1]), f64 = atoi(argv[a + 2]);
        const int slots = atoi(argv[a + 3]), split = atoi(argv[a + 4]);
        const int npad = (n + 1023) / 1024 * 1024, unit = f64 ? kSym64Unit : kSymUnit;
        const SymPlan p = make_sym_plan(n, npad, targets, f64 != 0, slots, split);
        const double warps = 4.0 * slots;
        double left = 0.0, longest = 0.0, over = 0.0;
        for (const SymItem &i : p.items) left += (double)i.nb * (i.j1 - i.j0);
        const double total = left;
        size_t at = 0;
        bool ok = true;
        int blocks = 0;
        for (size_t g = 0; g < p.rows.size(); ++g) {
            ok &= p.rows[g].first == (int)at;
            int j = -1;
            for (int k = 0; k < p.rows[g].items; ++k, ++at) {
                const SymItem &i = p.items[at];
                if (k == 0) {
                    ok &= i.ib0 == blocks && i.j0 == i.ib0 * targets;
                    blocks += i.nb;
                } else {
                    ok &= i.j0 == j && i.ib0 == p.items[at - 1].ib0 && i.nb == p.items[at - 1].nb;
                }
                ok &= i.j1 > i.j0 && i.j0 % unit == 0 && i.j1 % unit == 0;
                j = i.j1;
                const double len = (double)i.nb * (i.j1 - i.j0);
                // the shortest range is 256 sources (one unit with FP64)
                const double fair = left / (2.0 * warps), floor_ = (double)i.nb * (f64 ? unit : 256);
                over = std::max(over, len - std::max(fair, floor_));
                longest = std::max(longest, len);
                left -= len;
            }
            ok &= j == npad;
        }
        ok &= blocks == (n + targets - 1) / targets && at == p.items.size();
        ok &= p.part_doubles == p.items.size() * p.ki * 3 * (size_t)targets;
        std::priority_queue<double, std::vector<double>, std::greater<double>> ends;
        double last = 0.0;
        for (int w = 0; w < 4 * slots; ++w) ends.push(0.0);
        for (const SymItem &i : p.items) {
            const double end = ends.top() + (double)i.nb * (i.j1 - i.j0);
            ends.pop();
            ends.push(end);
            last = std::max(last, end);
        }
        printf("%zu %d %.6g %.6g %.6g\n", p.items.size(), (int)ok, over / total, longest / total,
               last * warps / total);
    }
}
"""


@pytest.fixture(scope="module")
def driver(tmp_path_factory):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no C++ compiler")
    d = tmp_path_factory.mktemp("plan")
    src = d / "plan.cpp"
    src.write_text(DRIVER)
    exe = str(d / "plan")
    subprocess.run([cxx, "-std=c++17", "-O1", "-Wall", "-I", build.CSRC, str(src), "-o", exe],
                   check=True)

    def plans(rows):
        args = [str(v) for r in rows for v in r]
        out = subprocess.run([exe, *args], check=True, capture_output=True, text=True).stdout
        return [(int(a), int(b), float(c), float(e), float(f)) for a, b, c, e, f in
                (line.split() for line in out.splitlines())]
    return plans


@pytest.mark.parametrize("n,targets,f64,slots", [
    (1 << 22, 512, 0, 456), (1 << 20, 512, 0, 456), ((1 << 20) - 77, 512, 0, 304),
    (1 << 20, 256, 0, 608), (100003, 512, 0, 456), (24001, 256, 0, 608), (14336, 256, 0, 456),
    (1, 256, 0, 456), (1 << 22, 32, 1, 304), (1 << 20, 32, 1, 304), (131072, 32, 1, 304),
    (16385, 32, 1, 304), (1, 32, 1, 304)])
def test_no_item_outlasts_the_pass_whatever_the_split(driver, n, targets, f64, slots):
    splits = (0, 1, 2, 3, 7, 64, 4096)
    got = driver([(n, targets, f64, slots, s) for s in splits])
    for s, (items, covered, over, longest, _) in zip(splits, got):
        assert covered == 1, s
        assert over <= 1e-12, s                 # of the pass's whole work
        assert longest <= got[0][3], s          # a split only shortens the ranges
        assert items >= got[0][0], s


@pytest.mark.parametrize("n,targets,slots", [
    (13001, 256, 608), (14336, 256, 456), (14336, 256, 608), (16385, 256, 456), (16385, 256, 608),
    (20481, 256, 456), (20481, 256, 608), (24576, 256, 608), (28673, 256, 608), (28673, 512, 456),
    (32768, 512, 456), (40001, 512, 456), (65536, 512, 456), (262144, 512, 456)])
def test_the_last_round_of_items_is_not_nearly_empty(driver, n, targets, slots):
    """Ranges of 256 sources whatever the number of warps left the last round of items of
    N = 20481 on 2432 warps half empty (1.36 times the even share), those of 128 sources that
    of N = 13001 (1.77).  A third over the even share is what one whole round of two to four
    costs at worst; the warps of a scheduler speed up when one of them has run out of work."""
    assert driver([(n, targets, 0, slots, 0)])[0][4] <= 4.0 / 3.0


FITS = r"""
#include <cstdio>
#include "pp_sym_plan.h"
int main()
{
    using ppk::sym_sums_fit;
    const size_t gb = size_t(1) << 30;
    printf("%d%d%d%d%d", sym_sums_fit(0, 0), sym_sums_fit(1, 3), sym_sums_fit(6 * gb, 24 * gb),
           sym_sums_fit(6 * gb + 1, 24 * gb), sym_sums_fit(29 * gb, 270 * gb));
}
"""


def test_partial_sums_take_a_quarter_of_the_free_memory_at_most(tmp_path):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no C++ compiler")
    (tmp_path / "fits.cpp").write_text(FITS)
    exe = str(tmp_path / "fits")
    subprocess.run([cxx, "-std=c++17", "-I", build.CSRC, str(tmp_path / "fits.cpp"), "-o", exe],
                   check=True)
    assert subprocess.run([exe], check=True, capture_output=True, text=True).stdout == "10101"

"""The CTAs of the narrow tree launch leave once the levels above their last
unit cannot use them (TreePlan::keep, compiled here with g++). Every unit must
still be taken whatever the grid and the order in which the CTAs run, no level
may be left with fewer CTAs than it has units, and the counts fall towards the
root."""
import os
import shutil
import subprocess

import numpy as np
import pytest

from kktgen import KKTPattern, make_grid

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2302_08656_gb300", "csrc")
CUDA_INC = "/usr/local/cuda/include"

SOURCE = """
#include "analysis.hpp"
#include "tree_plan.hpp"
#include <cstdio>
#include <cstdlib>
using namespace kktgb;
int main(int, char** a)
{
    std::FILE* f = std::fopen(a[1], "rb");
    int n = 0, nnz = 0;
    if (!f || std::fread(&n, 4, 1, f) != 1 || std::fread(&nnz, 4, 1, f) != 1) return 1;
    std::vector<int> rp(n + 1), ci(nnz);
    if (std::fread(rp.data(), 4, n + 1, f) != (size_t)n + 1 || std::fread(ci.data(), 4, nnz, f) != (size_t)nnz) return 1;
    AnalysisOptions opt;
    opt.max_pivots = std::atoi(a[2]);
    Analysis an;
    if (!analyze_pattern(n, rp.data(), ci.data(), opt, an).empty()) return 1;
    TreePlan tp;
    build_tree(an, 1 << 20, sizeof(double), tp);
    std::vector<int> lev(an.ns);
    for (int l = 0; l < an.n_levels; ++l)
        for (int t = an.level_ptr[l]; t < an.level_ptr[l + 1]; ++t) lev[an.level_fronts[t]] = l;
    for (size_t i = 0; i < tp.unit.size(); ++i) std::printf("0 %d %d\\n", lev[tp.fr[tp.unit[i].front].f], tp.keep[i]);
    for (size_t i = 0; i < tp.unit_fused.size(); ++i)
        std::printf("1 %d %d\\n", lev[tp.fr[tp.unit_fused[i].front].f], tp.keep_fused[i]);
    return 0;
}
"""


@pytest.fixture(scope="module")
def tool(tmp_path_factory):
    if shutil.which("g++") is None or not os.path.isdir(CUDA_INC):
        pytest.skip("g++ or the CUDA headers not available")
    d = tmp_path_factory.mktemp("keep")
    (d / "t.cpp").write_text(SOURCE)
    subprocess.run(["g++", "-O1", "-std=c++17", "-I", CSRC, "-I", CUDA_INC, str(d / "t.cpp"),
                    os.path.join(CSRC, "analysis.cpp"), os.path.join(CSRC, "tree_plan.cpp"), "-o", str(d / "t")],
                   check=True)
    return str(d / "t")


@pytest.mark.parametrize("buses,max_pivots", [(60, 16), (2003, 16), (500, 24)])
@pytest.mark.parametrize("order", [0, 1])
def test_every_unit_is_taken(tool, tmp_path, buses, max_pivots, order):
    pat = KKTPattern(make_grid(2, buses))
    with open(tmp_path / "in", "wb") as f:
        np.array([pat.n, pat.nnz], np.int32).tofile(f)
        np.asarray(pat.rowptr, np.int32).tofile(f)
        np.asarray(pat.colidx, np.int32).tofile(f)
    out = subprocess.run([tool, str(tmp_path / "in"), str(max_pivots)], check=True, capture_output=True, text=True)
    rows = np.array([line.split() for line in out.stdout.splitlines()], dtype=np.int64)
    level, keep = rows[rows[:, 0] == order][:, 1:].T
    assert np.all(np.diff(level) >= 0) and np.all(np.diff(keep) <= 0) and keep.min() >= 1
    width = np.bincount(level)
    for l in np.unique(level)[:-1]:
        assert keep[level == l].min() >= width[l + 1:].max()
    rng = np.random.default_rng(1)
    for grid in (1, 2, 9, 152):
        ticket, at = 0, {c: 1 << 30 for c in range(min(grid, level.size))}
        while at:                                              # a CTA at a time, in any order
            c = int(rng.choice(list(at)))
            if c >= at[c] or ticket == level.size:
                del at[c]
            else:
                at[c] = keep[ticket]
                ticket += 1
        assert ticket == level.size

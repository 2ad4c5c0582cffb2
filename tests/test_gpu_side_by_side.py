"""The front classes of a level side by side in a captured graph must not be
slower than the same kernels one after another: the times of two schedules of
one build on one device, each the median of many calls."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2302_08656_gb300 as K
from kktgen import KKTPattern, make_grid


def _median_ms(call, reps=9, n=20):
    out = []
    for _ in range(5):
        call()
    for _ in range(reps):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        torch.cuda.synchronize()
        a.record()
        for _ in range(n):
            call()
        b.record()
        torch.cuda.synchronize()
        out.append(a.elapsed_time(b) / n)
    return float(np.median(out))


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
def test_side_by_side_is_not_slower_than_one_after_another(precision):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    pat = KKTPattern(make_grid(100, 2003))                     # leaves of up to 8 and up to 16 rows, then the tree
    vals = torch.from_numpy(pat.values(pat.point(100, 0, 1e-3))).to("cuda:0")
    ms = {}
    for graphs in (True, False):
        s = K.KKTSolver(pat.rowptr, pat.colidx, pat.n_primal, precision=precision, graphs=graphs)
        ms[graphs] = _median_ms(lambda: s.refactor(vals))
        s.close()
    assert ms[True] <= 1.02 * ms[False], ms

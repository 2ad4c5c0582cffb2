"""The front classes of a level side by side in a captured graph must not be
slower than the same kernels one after another: the times of two schedules of
one build on one device, taken in turn."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2302_08656_gb300 as K
from kktgen import KKTPattern, make_grid


def best_ms(calls, reps=9, n=20):
    """The least time per call of each entry of calls, timed in turn."""
    best = {}
    for call in calls.values():
        for _ in range(5):
            call()
    for _ in range(reps):
        for key, call in calls.items():
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            torch.cuda.synchronize()
            a.record()
            for _ in range(n):
                call()
            b.record()
            torch.cuda.synchronize()
            best[key] = min(best.get(key, np.inf), a.elapsed_time(b) / n)
    return best


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
def test_side_by_side_is_not_slower_than_one_after_another(precision):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    pat = KKTPattern(make_grid(100, 2003))                     # leaves of up to 8 and up to 16 rows, then the tree
    vals = torch.from_numpy(pat.values(pat.point(100, 0, 1e-3))).to("cuda:0")
    side, turn = (K.KKTSolver(pat.rowptr, pat.colidx, pat.n_primal, precision=precision, graphs=g) for g in (True, False))
    ms = best_ms({"side by side": lambda: side.refactor(vals), "in turn": lambda: turn.refactor(vals)})
    side.close()
    turn.close()
    assert ms["side by side"] <= 1.02 * ms["in turn"], ms

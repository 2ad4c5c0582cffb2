"""kkt_residual with the backward error: its two kernels are counted and
profiled, the smallest system and restart length work, and an infinite or NaN
entry of x or of the right-hand side makes the backward error NaN."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2302_08656_gb300 as K
from kktgen import KKTPattern, make_grid


def _t(a):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return torch.from_numpy(np.ascontiguousarray(a, dtype=np.float64)).to("cuda:0")


@pytest.fixture(scope="module")
def system():
    pat = KKTPattern(make_grid(1, 60))
    v, b = _t(pat.values(pat.point(1, 0, 1e-2))), pat.rhs(1, 0)
    s = K.KKTSolver(pat.rowptr, pat.colidx, pat.n_primal)
    s.refactor(v)
    yield pat, s, b
    s.close()


def test_launches_are_counted_and_profiled(system):
    pat, s, b = system
    l0 = s.info().launches
    s.residual(_t(b), _t(np.ones(pat.n)))
    assert s.info().launches - l0 == 2
    s.set_profiling(True)
    s.residual(_t(b), _t(np.ones(pat.n)))
    stats = s.kernel_stats()
    s.set_profiling(False)
    assert stats["spmv_resid_kernel"][0] == 2


@pytest.mark.parametrize("bad", [np.inf, -np.inf, np.nan])
@pytest.mark.parametrize("where", ["x", "b"])
@pytest.mark.parametrize("row", [0, 37, -1])
def test_a_bad_entry_makes_the_backward_error_nan(system, bad, where, row):
    pat, s, b = system
    x, rhs = np.ones(pat.n), b.copy()
    (x if where == "x" else rhs)[row] = bad
    r, omega = s.residual(_t(rhs), _t(x))
    assert np.isnan(omega)                                     # NaN, or inf / inf
    assert not np.isfinite(r.cpu().numpy()[row])               # K has every diagonal entry
    _, again = s.residual(_t(b), _t(np.ones(pat.n)))
    assert np.isfinite(again)


def test_smallest_system_and_restart():
    s = K.KKTSolver(np.array([0, 1], np.int32), np.array([0], np.int32), 1, restart=1)
    s.refactor(_t([4.0]))
    r, omega = s.residual(_t([3.0]), _t([0.5]))
    assert r.item() == 1.0 and omega == 1.0 / (4.0 * 0.5 + 3.0)
    s.close()

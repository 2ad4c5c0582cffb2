"""Contexts that refactor at the same time share the SMs: sixteen systems on
forked streams (kkt_refactor_batched) against the same sixteen with the tops of
their trees in one launch (kkt_refactor_group), which keeps every SM full. Both
are timed in turn, one build on one device; the forked launches
took 1.12 to 1.23 times as long as the group where several CTAs of the narrow
tree launch fit on an SM, 1.9 times where one filled it."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2302_08656_gb300 as K
from kktgen import KKTPattern, make_grid
from test_gpu_side_by_side import best_ms


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
def test_forked_streams_keep_up_with_the_group_launch(precision):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    solvers, vals = [], []
    for i in range(16):
        pat = KKTPattern(make_grid(100 + i, 2003 + i))
        solvers.append(K.KKTSolver(pat.rowptr, pat.colidx, pat.n_primal, precision=precision))
        vals.append(torch.from_numpy(pat.values(pat.point(100 + i, 0, 1e-3))).to("cuda:0"))
    group = K.KKTGroup(solvers)
    ms = best_ms({"group": lambda: group.refactor(vals), "forked": lambda: K.refactor_batched(solvers, vals)})
    group.close()
    for s in solvers:
        s.close()
    assert ms["forked"] <= 1.5 * ms["group"], ms

"""The forward step of the tree part inside kkt_refactor_refine. With mini
fronts of at most 32 rows (max_pivots <= 16) it runs inside the factorization
units (ti, 0), a lane per row; with larger ones it runs as units of its own.
Both must equal the separate refactorization and solve bit for bit, and so
must the gather of the children's blocks by column, which the first
factorization uses as well: fronts with one child and with dozens, one tile and
many, both precisions, one instance and several."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2302_08656_gb300 as K
from kktgen import KKTPattern, make_grid


@pytest.fixture(scope="module", params=[(60, 1), (1203, 5)], ids=["60", "1203"])
def pattern(request):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    buses, seed = request.param
    return KKTPattern(make_grid(seed, buses))


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("max_pivots", [3, 16, 24])
@pytest.mark.parametrize("count", [1, 3])
def test_fused_forward_equals_separate_calls(pattern, precision, max_pivots, count):
    pat, dev = pattern, torch.device("cuda:0")
    vals = torch.from_numpy(np.concatenate([pat.values(pat.point(2, i, 1e-3)) for i in range(count)])).to(dev)
    rhs = torch.from_numpy(np.concatenate([pat.rhs(2, i) for i in range(count)])).to(dev)
    out = []
    # a tolerance that any first solve meets: x is the solve itself
    for tmf in (1 << 20, 0):
        s = K.KKTSolver(pat.rowptr, pat.colidx, pat.n_primal, count=count, precision=precision,
                        max_pivots=max_pivots, tree_min_fronts=tmf)
        assert (s.plan()["tree_levels"] > 0) == (tmf > 0)
        for _ in range(2):                                     # the second call replays the captured graphs
            x, _ = s.refactor_refine(vals, rhs, tol=1.0)
            out.append(x.cpu().numpy())
        s.refactor(vals)
        out.append(s.solve(rhs).cpu().numpy())
        s.close()
    for x in out[1:]:
        assert np.array_equal(out[0], x)

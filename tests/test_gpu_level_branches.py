"""The front classes of a level run side by side in the captured graphs and one
after another when launched directly: the same bits, with every class present
(leaves of up to 8 and 16 rows, warp, CTA and panel fronts), fused and in
separate calls."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2302_08656_gb300 as K
from kktgen import KKTPattern, make_grid


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("buses,count", [(411, 3), (6011, 1)])
def test_graphs_equal_direct_launches(precision, buses, count):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    pat, dev = KKTPattern(make_grid(8, buses)), torch.device("cuda:0")
    vals = torch.from_numpy(np.concatenate([pat.values(pat.point(4, i, 1e-3)) for i in range(count)])).to(dev)
    rhs = torch.from_numpy(np.concatenate([pat.rhs(4, i) for i in range(count)])).to(dev)
    out = []
    for graphs in (False, True):
        s = K.KKTSolver(pat.rowptr, pat.colidx, pat.n_primal, count=count, precision=precision, tree_min_fronts=0,
                        graphs=graphs)
        for _ in range(2):                                     # the second call replays the graphs
            s.refactor(vals)
            out.append(s.solve(rhs).cpu().numpy())
            x, _ = s.refactor_refine(vals, rhs, tol=1.0)       # any first solve meets it
            out.append(x.cpu().numpy())
        s.close()
    for x in out[1:]:
        assert np.array_equal(out[0], x)

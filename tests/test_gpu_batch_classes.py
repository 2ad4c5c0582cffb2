"""The front class of a level counts the fronts of all instances of a batch:
the same system with one instance (CTA kernels on its narrow levels) and with
many (warp kernels) must give the same bits, level launched and by the tree
kernels, fused and in separate calls."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2302_08656_gb300 as K
from kktgen import KKTPattern, make_grid


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("count", [2, 31])
@pytest.mark.parametrize("tree_min_fronts", [0, 2432])
def test_batch_equals_its_instances(precision, count, tree_min_fronts):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    pat, dev = KKTPattern(make_grid(4, 411)), torch.device("cuda:0")
    vals = [torch.from_numpy(pat.values(pat.point(3, i, 1e-2))).to(dev) for i in range(count)]
    rhs = [torch.from_numpy(pat.rhs(3, i)).to(dev) for i in range(count)]
    opts = dict(precision=precision, tree_min_fronts=tree_min_fronts)
    many = K.KKTSolver(pat.rowptr, pat.colidx, pat.n_primal, count=count, **opts)
    one = K.KKTSolver(pat.rowptr, pat.colidx, pat.n_primal, **opts)
    v, b = torch.cat(vals), torch.cat(rhs)
    x, _ = many.refactor_refine(v, b, tol=1.0)                 # any first solve meets it
    x = x.cpu().numpy().reshape(count, -1)
    many.refactor(v)
    y = many.solve(b).cpu().numpy().reshape(count, -1)
    for i in (0, count - 1):
        z, _ = one.refactor_refine(vals[i], rhs[i], tol=1.0)
        z = z.cpu().numpy()
        assert np.array_equal(x[i], z) and np.array_equal(y[i], z)
    many.close()
    one.close()

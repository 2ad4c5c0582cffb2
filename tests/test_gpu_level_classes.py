"""The systems on which the captured graphs are compared with direct launches
(test_gpu_level_branches.py) hold every front class that a level can run side by
side: the kernels that a refactorization launches, by name."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2302_08656_gb300 as K
from kktgen import KKTPattern, make_grid


def test_every_front_class_runs():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    launched = {}
    for buses, count in ((411, 3), (6011, 1)):
        pat = KKTPattern(make_grid(8, buses))
        vals = np.concatenate([pat.values(pat.point(4, i, 1e-3)) for i in range(count)])
        s = K.KKTSolver(pat.rowptr, pat.colidx, pat.n_primal, count=count, tree_min_fronts=0, graphs=False)
        s.set_profiling(True)
        s.refactor(torch.from_numpy(vals).to("cuda:0"))
        for name, (launches, _) in s.kernel_stats().items():
            launched[name] = max(launched.get(name, 0), launches)
        s.close()
    # every childless front is on the lowest level: two launches are leaves of both sizes there
    assert launched["front_leaf_kernel"] == 2
    for name in ("front_warp_kernel", "front_cta_kernel", "front_panel_kernel", "schur_tile_kernel"):
        assert launched.get(name, 0) > 0, launched

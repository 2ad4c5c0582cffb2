"""The pivot rule of every FP64 factorization kernel at its edges: entries just
below, at and just above the static-pivot floor (also with the floor's own high
word), zero, and both ends of the range of the fast reciprocal. Blocks of one
special pivot each, unscaled (no Ruiz iterations): U(p, p) must be the entry or
sign(entry) * floor, L(p + 1, p) the entry below it times the reciprocal of
that pivot, and the count of events exact. The shapes take the leaf (8 and 16
rows), warp, CTA and panel kernels, and both forms of the tree kernel."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2302_08656_gb300 as K

FLOOR = 1.3e-6                                                     # a mantissa with a low word
TINY, HUGE = 2.0 ** -1000, 2.0 ** 1001
# (static_pivot_eps, entry beside the pivot, special pivots): the largest entry of K is 1, 1 and HUGE
EDGES = {
    "floor": (FLOOR, 2.0 ** -12, [np.nextafter(FLOOR, 0), FLOOR, np.nextafter(FLOOR, 1), FLOOR * (1 + 2.0 ** -30),
                                  FLOOR * (1 - 2.0 ** -30), FLOOR / 2, FLOOR * 2, 0.0, 5e-324, 0.75]),
    "small": (2.0 ** -1022, 2.0 ** -700, [TINY / 2, np.nextafter(TINY, 0), TINY, np.nextafter(TINY, 1), 2 * TINY]),
    "large": (2.0 ** -1010, 1.0, [HUGE, np.nextafter(HUGE, 0), HUGE / 2, np.nextafter(HUGE / 2, 0)]),
}
# kernel: rows of a block, number of blocks, max_pivots, tree_min_fronts
SHAPES = {
    "front_leaf_kernel 8": (2, 700, 16, 0),
    "front_leaf_kernel 16": (12, 700, 16, 0),
    "front_warp_kernel": (18, 700, 32, 0),
    "front_cta_kernel": (18, 40, 32, 0),
    "front_panel_kernel": (100, 30, 16, 0),
    "tree_factor_kernel narrow": (2, 40, 16, 1 << 20),
    "tree_factor_kernel wide": (2, 700, 16, 1 << 20),
    "tree_factor_kernel tiles": (100, 30, 16, 1 << 20),
    "tree_factor_kernel large": (40, 30, 64, 1 << 20),
}


@pytest.mark.parametrize("shape", sorted(SHAPES))
@pytest.mark.parametrize("edge", sorted(EDGES))
def test_pivots_at_the_edges(shape, edge):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    size, blocks, max_pivots, tree_min_fronts = SHAPES[shape]
    eps, beside, entries = EDGES[edge]
    entries = np.array(entries + [-e for e in entries])
    first = size * np.arange(blocks)
    p = entries[np.arange(blocks) % entries.size]
    block = np.eye(size)
    block[0, 1] = block[1, 0] = beside
    vals = np.tile(block, (blocks, 1, 1))
    vals[:, 0, 0] = p
    floor = eps * np.abs(vals).max()
    n = size * blocks
    rp = (size * np.arange(n + 1)).astype(np.int32)
    ci = (np.repeat(first, size * size) + np.tile(np.arange(size), n)).astype(np.int32)
    dev = torch.device("cuda:0")
    s = K.KKTSolver(rp, ci, n, user_perm=np.arange(n), static_pivot_eps=eps, ruiz_iters=0, max_pivots=max_pivots,
                    tree_min_fronts=tree_min_fronts)
    s.set_profiling(True)
    s.refactor(torch.from_numpy(vals.reshape(-1)).to(dev))
    assert shape.split()[0] in s.kernel_stats()
    s.set_profiling(False)
    below = np.abs(p) < floor
    want = np.where(below, np.where(p < 0, -floor, floor), p)
    rcp = K.debug_pivot_rcp(torch.from_numpy(want).to(dev)).cpu().numpy()
    lr, lc, lv, ur, uc, uv = s.export_factors()
    u = dict(zip(ur[ur == uc], uv[ur == uc]))
    sel = (lr == lc + 1) & (lc % size == 0)
    low = dict(zip(lc[sel], lv[sel]))
    assert np.array_equal([u[f] for f in first], want)
    assert np.array_equal([low[f] for f in first], beside * rcp)
    assert s.info().n_perturbed == below.sum() and s.info().status == 0
    s.close()

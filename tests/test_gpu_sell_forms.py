"""The two forms of the passes over the sliced copy of K, on either side of
the boundary (8,192 slices over all instances of a batch): up to it a row's
long slices are cut into segments, beyond it a warp takes a whole slice.
Equilibration (with a subnormal entry as well) must equal the oracle's bit for
bit on both sides, the residual sums in CSR order within one rounding per term,
and every instance of a batch its own solver."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import oracle as O
import paper_2302_08656_gb300 as K
from kktgen import KKTPattern, make_grid
from test_gpu_sell_segments import _arrow

SEGMENTED = 8192                                                   # slices of 32 rows, all instances together


def _t(a):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return torch.from_numpy(np.ascontiguousarray(a, dtype=np.float64)).to("cuda:0")


def _check_residual(s, rp, ci, vals, seed):
    """r and omega of instance 0 against sums in extended precision."""
    n = len(rp) - 1
    rng = np.random.default_rng(seed)
    b, x = rng.normal(size=n), rng.normal(size=n)
    r, omega = s.residual(_t(b), _t(x))
    rows = np.repeat(np.arange(n), np.diff(rp))
    term = vals.astype(np.longdouble) * x[ci]
    ref = np.asarray(b, np.longdouble).copy()
    np.subtract.at(ref, rows, term)
    absrow, krow = np.zeros(n), np.zeros(n)
    np.add.at(absrow, rows, np.abs(term).astype(float))
    np.add.at(krow, rows, np.abs(vals))
    u, lens, r = 2.0 ** -53, np.diff(rp), r.cpu().numpy()
    # one rounding per term and one of the difference on either side of the exact value
    assert np.all(np.abs(r - ref) <= (lens + 2) * u * (absrow + np.abs(b)))
    want = np.abs(r).max() / (krow.max() * np.abs(x).max() + np.abs(b).max())
    assert abs(omega - want) <= (lens.max() + 8) * u * want


@pytest.mark.parametrize("over", [0, 1], ids=["segments", "whole"])
@pytest.mark.parametrize("n,widths", [(33, [8, 9, 16, 17, 30]), (321, [63, 64, 65]), (321, [1, 2, 129, 200])], ids=str)
def test_rows_of_many_lengths(n, widths, over):
    rp, ci, vals = _arrow(n, [min(w, n - len(widths)) for w in widths], 5)
    count = SEGMENTED // ((n + 31) // 32) + over
    scale = np.ldexp(1.0, np.arange(count) % 7)                    # instance 0 as it is
    s = K.KKTSolver(rp, ci, n, count=count)
    s.refactor(_t((scale[:, None] * vals[None, :]).reshape(-1)))
    assert np.array_equal(s.scaling(), O.ruiz(rp, ci, vals, 10)[0])
    _check_residual(s, rp, ci, vals, 6)
    s.close()


@pytest.fixture(scope="module")
def pattern():
    return KKTPattern(make_grid(3, 300))


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
def test_whole_slices_equal_segments_instance_by_instance(pattern, precision):
    """A batch beyond the boundary against one solver (segmented) per instance."""
    pat = pattern
    count = SEGMENTED // ((pat.n + 31) // 32) + 1
    vals = np.stack([pat.values(pat.point(3, i, 10.0 ** -(1 + i % 4))) for i in range(count)])
    rhs = np.stack([pat.rhs(3, i) for i in range(count)])
    off = pat.rowptr[:-1][np.diff(pat.rowptr) > 8][0] + 1           # an off-diagonal entry and its mirror
    i, j = int(np.searchsorted(pat.rowptr, off, side="right")) - 1, int(pat.colidx[off])
    mirror = pat.rowptr[j] + int(np.searchsorted(pat.colidx[pat.rowptr[j]:pat.rowptr[j + 1]], i))
    assert i != j and pat.colidx[mirror] == i
    vals[0, [off, mirror]] = 1e-310                                # instance 0 takes the subnormal path
    many = K.KKTSolver(pat.rowptr, pat.colidx, pat.n_primal, count=count, precision=precision)
    one = K.KKTSolver(pat.rowptr, pat.colidx, pat.n_primal, precision=precision)
    x, infos = many.refactor_refine(_t(vals.reshape(-1)), _t(rhs.reshape(-1)), tol=1.0)   # any first solve meets it
    x = x.cpu().numpy().reshape(count, -1)
    for k in (0, 1, count // 2, count - 1):
        z, info = one.refactor_refine(_t(vals[k]), _t(rhs[k]), tol=1.0)
        assert np.array_equal(x[k], z.cpu().numpy())
        assert infos[k].backward_err == info.backward_err and infos[k].n_perturbed == info.n_perturbed
    assert np.array_equal(many.scaling(), O.ruiz(pat.rowptr, pat.colidx, vals[0], 10)[0])
    _check_residual(many, pat.rowptr, pat.colidx, vals[0], 7)
    many.close()
    one.close()


@pytest.mark.parametrize("bad", [np.inf, np.nan])
def test_bad_entries_stay_in_their_instance(pattern, bad):
    """An infinite or NaN entry of one instance: that instance's backward error is not finite, the others' x unchanged."""
    pat = pattern
    count = SEGMENTED // ((pat.n + 31) // 32) + 1
    vals = np.stack([pat.values(pat.point(3, i, 1e-2)) for i in range(count)])
    rhs = np.stack([pat.rhs(3, i) for i in range(count)])
    many = K.KKTSolver(pat.rowptr, pat.colidx, pat.n_primal, count=count)
    many.refactor(_t(vals.reshape(-1)))
    clean = many.solve(_t(rhs.reshape(-1))).cpu().numpy().reshape(count, -1)
    vals[5, pat.rowptr[7]] = bad
    many.refactor(_t(vals.reshape(-1)))
    omega = torch.empty(count, dtype=torch.float64).pin_memory()
    x = torch.empty(count * pat.n, dtype=torch.float64, device="cuda:0")
    many.solve_checked(_t(rhs.reshape(-1)), x, omega)
    torch.cuda.synchronize()
    om, x = omega.numpy(), x.cpu().numpy().reshape(count, -1)
    rest = np.arange(count) != 5
    assert not np.isfinite(om[5]) and np.all(om[rest] <= 1e-10) and np.array_equal(x[rest], clean[rest])
    many.close()

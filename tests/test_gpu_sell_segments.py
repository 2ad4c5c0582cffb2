"""Passes over the sliced copy of K on rows of every kind of length: one round
of slots, a segment's edge, several segments, more slots than a block's warps
take in one round. Equilibration equals the oracle's bit for bit, ||K||_inf and
the residual equal sums in CSR order (both of one rounding per term)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import oracle as O
import paper_2302_08656_gb300 as K


def _arrow(n, widths, seed):
    """Symmetric pattern of size n: a diagonal, and row r of widths[r] entries with its mirror column."""
    rng = np.random.default_rng(seed)
    rows = [{i} for i in range(n)]
    for r, w in enumerate(widths):
        for c in range(n - w + 1, n):
            rows[r].add(c)
            rows[c].add(r)
    rp = np.cumsum([0] + [len(s) for s in rows]).astype(np.int32)
    ci = np.concatenate([np.sort(np.fromiter(s, np.int32)) for s in rows]).astype(np.int32)
    v = {}
    vals = np.empty(ci.size)
    for i in range(n):
        for p in range(rp[i], rp[i + 1]):
            key = (min(i, ci[p]), max(i, ci[p]))
            if key not in v:
                v[key] = rng.normal() * 10.0 ** rng.uniform(-6, 6) + (1e7 if i == ci[p] else 0.0)
            vals[p] = v[key]
    return rp, ci, vals


@pytest.mark.parametrize("widths", [[8, 9, 16, 17], [63, 64, 65], [1, 2, 129, 200], [24] * 40], ids=str)
@pytest.mark.parametrize("n", [33, 321])
def test_rows_of_many_lengths(widths, n):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    widths = [min(w, n - len(widths)) for w in widths[:n // 2]]
    rp, ci, vals = _arrow(n, widths, 5)
    rng = np.random.default_rng(6)
    b, x = rng.normal(size=n), rng.normal(size=n)
    dev = torch.device("cuda:0")
    s = K.KKTSolver(rp, ci, n)
    s.refactor(torch.from_numpy(vals).to(dev))
    d, _ = O.ruiz(rp, ci, vals, 10)
    assert np.array_equal(s.scaling(), d)
    r, omega = s.residual(torch.from_numpy(b).to(dev), torch.from_numpy(x).to(dev))
    r = r.cpu().numpy()
    # one rounding per term and one of the difference on either side of the exact value
    lens = np.diff(rp)
    absrow = np.array([np.abs(vals[rp[i]:rp[i + 1]] * x[ci[rp[i]:rp[i + 1]]]).sum() for i in range(n)])
    ref = np.array([b[i] - np.dot(vals[rp[i]:rp[i + 1]].astype(np.longdouble), x[ci[rp[i]:rp[i + 1]]])
                    for i in range(n)])
    u = 2.0 ** -53
    assert np.all(np.abs(r - ref) <= (lens + 2) * u * (absrow + np.abs(b)))
    knorm = max(np.abs(vals[rp[i]:rp[i + 1]]).sum() for i in range(n))
    want = np.abs(r).max() / (knorm * np.abs(x).max() + np.abs(b).max())
    assert abs(omega - want) <= (lens.max() + 8) * u * want
    s.close()

"""The FP64 judge (nb_direct_sum) at the edges of its target and source split,
against numpy's FP64 sum: odd target counts, clusters of 1 to 8 blocks, fewer
sources than threads, coincident points without
softening, and separations whose squares leave the range of the reciprocal
square root's fast path.  FP64 sums in another order: 1e-12 of sum |a_ij|.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)


def _check(pos, mass, eps, targets):
    import paper_0909_0541_gb300 as nb
    dev = torch.device("cuda")
    t = None if targets is None else torch.from_numpy(np.asarray(targets, np.int64)).to(dev)
    a, p = nb.direct_sum(torch.from_numpy(pos).to(dev), torch.from_numpy(mass).to(dev), eps, t)
    a, p = a.cpu().numpy(), p.cpu().numpy()
    rows = np.arange(len(pos)) if targets is None else np.asarray(targets)
    m = mass.astype(np.float64)
    with np.errstate(over="ignore", divide="ignore", invalid="ignore"):
        for k in (range(len(rows)) if len(rows) <= 200 else
                  np.random.default_rng(1).choice(len(rows), 200, replace=False)):
            i = rows[k]
            d = pos - pos[i]
            r2 = (d * d).sum(1) + eps * eps
            ok = (r2 > 0) & (np.arange(len(pos)) != i)
            ri = np.where(ok, 1.0 / np.sqrt(np.where(ok, r2, 1.0)), 0.0)
            w = (m * ri * ri * ri)[:, None] * d
            tol = 1e-12 * np.abs(w).sum(0) + 1e-300
            assert np.all(np.abs(a[k] - w.sum(0)) <= tol), (i, a[k], w.sum(0))
            assert abs(p[k] + (m * ri).sum()) <= 1e-12 * (m * ri).sum() + 1e-300


@pytest.mark.parametrize("n,nt", [(1, 1), (2, 2), (255, 7), (257, 9), (1000, 33), (4096, 3),
                                  (16385, 1), (9000, 301), (9000, 1300), (3001, None)])
def test_splits(n, nt):
    rng = np.random.default_rng(n)
    pos = rng.normal(size=(n, 3))
    mass = rng.uniform(0.5, 1.5, n).astype(np.float32) / n
    t = None if nt is None else rng.integers(0, n, nt)
    _check(pos, mass, 1.0 / 64, t)


@pytest.mark.parametrize("scale", [1.0, 1e-95, 1e-19, 1e18, 1e100, 1e148, 1e160])
def test_coincident_points_and_extreme_separations(scale):
    rng = np.random.default_rng(9)
    pos = rng.normal(size=(600, 3)) * scale
    pos[100:110] = pos[5]
    mass = np.full(600, 1e-3, np.float32)
    _check(pos, mass, 0.0, [0, 5, 100, 109, 599])

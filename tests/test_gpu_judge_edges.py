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


@pytest.mark.parametrize("more", [-1, 0, 1, 2])
@pytest.mark.parametrize("n", [300, 5000])
def test_one_and_two_targets_per_block(n, more):
    """Either side of one target per SM, where a block takes a second one."""
    rng = np.random.default_rng(n + more)
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    mass = rng.uniform(0.5, 1.5, n).astype(np.float32) / n
    _check(rng.normal(size=(n, 3)), mass, 1.0 / 64, rng.integers(0, n, sms + more))


@pytest.mark.parametrize("scale", [1.0, 1e-95, 1e-19, 1e18, 1e100, 1e148, 1e160])
def test_coincident_points_and_extreme_separations(scale):
    rng = np.random.default_rng(9)
    pos = rng.normal(size=(600, 3)) * scale
    pos[100:110] = pos[5]
    mass = np.full(600, 1e-3, np.float32)
    _check(pos, mass, 0.0, [0, 5, 100, 109, 599])


def test_left_out_pairs_are_left_out_whatever_they_hold():
    """The target itself and coincident pairs (eps = 0) add nothing, also where
    their mass or a coordinate is not finite: the sums of the other pairs."""
    import paper_0909_0541_gb300 as nb
    rng = np.random.default_rng(4)
    n = 700
    dev = torch.device("cuda")
    for case in ("mass", "position"):
        pos, mass = rng.normal(size=(n, 3)), rng.uniform(0.5, 1.5, n).astype(np.float32) / n
        i = 10
        if case == "mass":
            pos[20:23] = pos[i]
            mass[20], mass[21], mass[i] = np.inf, np.nan, np.inf
        else:
            pos[i, 1] = np.inf
        a, p = nb.direct_sum(torch.from_numpy(pos).to(dev), torch.from_numpy(mass).to(dev), 0.0,
                             torch.tensor([i], device=dev))
        a, p = a.cpu().numpy()[0], p.cpu().numpy()[0]
        m = mass.astype(np.float64)
        with np.errstate(all="ignore"):
            d = pos - pos[i]
            r2 = (d * d).sum(1)
            ok = (np.arange(n) != i) & (r2 != 0)
            ri = 1.0 / np.sqrt(r2[ok])
            want = ((m[ok] * ri * ri * ri)[:, None] * d[ok]).sum(0)
            wp = -(m[ok] * ri).sum()
        # FP64 sums in another order; an infinite position leaves 0 x inf = NaN
        # along its axis and 0 elsewhere
        assert np.allclose(a, want, rtol=1e-11, atol=1e-12, equal_nan=True), case
        assert np.isfinite(wp) and abs(p - wp) <= 1e-12 * abs(wp), case
    one, _ = nb.direct_sum(torch.full((1, 3), np.inf, dtype=torch.float64, device=dev),
                           torch.ones(1, device=dev), 0.0)
    assert torch.equal(one, torch.zeros_like(one))

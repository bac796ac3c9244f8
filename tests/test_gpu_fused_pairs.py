"""The fused pass where two neighbouring work items share a walk (items of 32
and of 16 targets, large groups) and just outside that range: the same bits as
the list path in every precision, with and without softening, for groups with
even and odd numbers of full items and every remainder, and for a forest.  The
interaction counts are those of the list path.
"""
import numpy as np
import pytest

import nbsynth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)


def _equal(ctx, n, theta, n_crit, eps, precision):
    dev = torch.device("cuda")
    out = []
    for fused in (False, True):
        acc = torch.full((n, 3), np.nan, dtype=torch.float32, device=dev)
        pot = torch.full((n,), np.nan, dtype=torch.float32, device=dev)
        if fused:
            ctx.forces_fused(theta, n_crit, eps, acc, pot, precision)
        else:
            ctx.walk_groups(theta, n_crit)
            ctx.forces(eps, acc, pot, precision)
        out.append((acc, pot, ctx.stats()))
    (a, p, s), (b, q, t) = out
    assert torch.equal(a, b) and torch.equal(p, q)
    assert bool(torch.isfinite(a).all())
    for k in ("n_groups", "list_entries", "max_list", "n_pp", "n_pc"):
        assert s[k] == t[k], k


@pytest.mark.parametrize("precision", ["fp32", "fp32_comp", "fp64acc"])
@pytest.mark.parametrize("n,n_crit", [(24400, 256), (32768, 301), (60001, 512), (70000, 1000),
                                      (70000, 100000), (40000, 256), (300000, 128)])
def test_equal_to_lists(n, n_crit, precision):
    import paper_0909_0541_gb300 as nb
    ps = nbsynth.halo_mix(n, n % 97, n_halos=15)
    dev = torch.device("cuda")
    ctx = nb.NBody(n)
    ctx.build_tree(torch.from_numpy(ps.pos).to(dev), torch.from_numpy(ps.mass).to(dev))
    for eps in (1e-3, 0.0):
        if precision == "fp64acc" and n_crit > 1000:
            continue
        _equal(ctx, n, 0.7, n_crit, eps, precision)
    ctx.close()


def test_forest():
    import paper_0909_0541_gb300 as nb
    systems = [nbsynth.plummer(n, n) for n in (30000, 257, 20000, 33, 15000, 1)]
    off = np.r_[0, np.cumsum([s.n for s in systems])].astype(np.int64)
    pos = np.concatenate([s.pos for s in systems])
    mass = np.concatenate([s.mass for s in systems])
    dev = torch.device("cuda")
    ctx = nb.NBody(len(pos), max_systems=len(systems))
    ctx.build_tree_batched(torch.from_numpy(pos).to(dev), torch.from_numpy(mass).to(dev),
                           torch.from_numpy(off).to(dev))
    _equal(ctx, len(pos), 0.7, 512, 1e-3, "fp32")
    ctx.close()

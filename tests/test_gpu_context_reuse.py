"""One context used again: a walk that outgrows the storage of the one before.
A walk that fails for lack of storage is repeated once, after the storage has
grown: one more launch than a walk that fits.  Walks that failed are not in
n_pp_total / n_pc_total.  The lists are those of a fresh context.
"""
import numpy as np
import pytest

import nbsynth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)


def _set(n, seed, **kw):
    import paper_0909_0541_gb300 as nb
    ps = nbsynth.plummer(n, seed)
    dev = torch.device("cuda")
    x, m = torch.from_numpy(ps.pos).to(dev), torch.from_numpy(ps.mass).to(dev)
    ctx = nb.NBody(n, **kw)
    ctx.build_tree(x, m)
    return ctx, x, m


def _walk(ctx, theta, n_crit):
    """(launches, growth of the total counts, the walk's own counts)"""
    a = ctx.stats()
    ctx.get_timing()
    ctx.walk_groups(theta, n_crit)
    launches = ctx.get_timing()["launches"]
    b = ctx.stats()
    return (launches, (b["n_pp_total"] - a["n_pp_total"], b["n_pc_total"] - a["n_pc_total"]),
            (b["n_pp"], b["n_pc"]))


def _same_lists(ctx, x, m, theta, n_crit):
    import paper_0909_0541_gb300 as nb
    one = nb.NBody(len(x))
    one.build_tree(x, m)
    one.walk_groups(theta, n_crit)
    a, b = ctx.copy_lists(with_xm=True), one.copy_lists(with_xm=True)
    one.close()
    assert all(np.array_equal(a[k], b[k]) for k in ("offsets", "entries", "xm"))


@pytest.mark.parametrize("n", [3000, 9000])
@pytest.mark.parametrize("first,then,extra", [
    ((1.0, 64), (0.3, 64), 1),     # lists longer than a slot
    ((0.6, 512), (0.6, 8), 1),     # more groups than the storage holds
    ((1.0, 512), (0.0, 512), 2),   # frontiers wider than the queues, and long lists
])
def test_walk_that_outgrows_its_storage(n, first, then, extra):
    ctx, x, m = _set(n, 5)
    ctx.walk_groups(*first)
    plain, total, own = _walk(ctx, *first)
    assert total == own
    launches, total, own = _walk(ctx, *then)
    assert plain <= launches <= plain + extra
    assert total == own
    _same_lists(ctx, x, m, *then)
    assert _walk(ctx, *then)[0] == plain
    ctx.close()


def test_fixed_list_capacity():
    """A caller's own slot size is never changed: more groups take more
    storage, a list longer than the slot is NB_ERR_CAPACITY."""
    import paper_0909_0541_gb300 as nb
    ctx, x, m = _set(4000, 6, list_capacity=1024)
    ctx.walk_groups(1.0, 256)
    ctx.walk_groups(1.0, 16)
    assert ctx.stats()["list_capacity"] == 1024
    _same_lists(ctx, x, m, 1.0, 16)
    with pytest.raises(nb.NBError) as e:
        ctx.walk_groups(0.1, 16)
    assert e.value.code == -3
    ctx.walk_groups(1.0, 16)
    _same_lists(ctx, x, m, 1.0, 16)
    ctx.close()


@pytest.mark.parametrize("call", ["forces_fused", "walk_forces"])
def test_repeated_passes_count_once(call):
    """The overlapped pass that falls back, and the fused pass whose frontier
    queues grow: counted once, the forces those of separate calls."""
    n = 9000
    ctx, x, m = _set(n, 7)
    ctx.walk_groups(1.0, 512)
    acc, ref = (torch.empty((n, 3), dtype=torch.float32, device=x.device) for _ in range(2))
    a = ctx.stats()
    getattr(ctx, call)(0.0, 512, 1e-3, acc)
    b = ctx.stats()
    assert b["n_pp_total"] - a["n_pp_total"] == b["n_pp"]
    assert b["n_pc_total"] - a["n_pc_total"] == b["n_pc"]
    ctx.walk_groups(0.0, 512)
    ctx.forces(1e-3, ref)
    assert torch.equal(acc, ref)
    ctx.close()

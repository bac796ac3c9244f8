"""The (system, key) order of a batch where the system number rides in the
sorted values: one digit up to 256 systems, two beyond, odd sizes, and equal
keys (coincident particles keep the caller's order).  Every system's slots
must be the stable key order of its own rows, with the keys that system's
tree gets when it is built alone.  The same where index and system do not fit
32 bits and a second sort orders the systems, by two digits up to 65,536
systems and by four beyond.
"""
import numpy as np
import pytest

import nbsynth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)


@pytest.mark.parametrize("nsys,lo,hi", [(2, 1, 5000), (255, 1, 60), (256, 3, 40), (257, 1, 50),
                                        (700, 1, 30)])
def test_order_is_stable_by_system_and_key(nsys, lo, hi):
    import paper_0909_0541_gb300 as nb
    rng = np.random.default_rng(nsys)
    size = rng.integers(lo, hi + 1, nsys)
    off = np.concatenate([[0], np.cumsum(size)]).astype(np.int64)
    n = int(off[-1])
    pos = nbsynth.uniform_cube(n, 17 + nsys).pos * rng.uniform(0.1, 10.0)
    for s in range(0, nsys, 3):            # coincident particles in some systems
        if size[s] > 3:
            pos[off[s] + 1:off[s] + 3] = pos[off[s]]
    dev = torch.device("cuda")
    x = torch.from_numpy(pos).to(dev)
    m = torch.full((n,), 1.0 / n, dtype=torch.float32, device=dev)
    ctx = nb.NBody(n, max_systems=nsys)
    ctx.build_tree_batched(x, m, torch.from_numpy(off).to(dev))
    t = ctx.copy_tree()
    keys, perm = t["keys"], t["perm"]
    assert np.array_equal(np.sort(perm), np.arange(n))
    for s in range(nsys):
        a, b = off[s], off[s + 1]
        p, k = perm[a:b], keys[a:b]
        assert p.min() >= a and p.max() < b, s
        assert np.all((k[1:] > k[:-1]) | ((k[1:] == k[:-1]) & (p[1:] > p[:-1]))), s
    for s in (0, nsys // 2, nsys - 1):
        a, b = off[s], off[s + 1]
        one = nb.NBody(int(b - a))
        one.build_tree(x[a:b].contiguous(), m[a:b].contiguous())
        o = one.copy_tree()
        assert np.array_equal(o["keys"], keys[a:b]) and np.array_equal(o["perm"] + a, perm[a:b])
        one.close()
    ctx.close()


@pytest.mark.parametrize("nsys,lo,hi", [(33000, 1, 3), (65536, 1, 2), (65537, 1, 2),
                                        (140000, 1, 2)])
def test_order_by_a_second_sort(nsys, lo, hi):
    test_order_is_stable_by_system_and_key(nsys, lo, hi)


def test_forces_of_more_systems_than_two_digits_hold():
    """Pairs: each particle's acceleration is its partner's pull alone."""
    import paper_0909_0541_gb300 as nb
    nsys = 70_000
    pos = nbsynth.uniform_cube(2 * nsys, 5).pos
    dev = torch.device("cuda")
    x = torch.from_numpy(pos).to(dev)
    m = torch.full((2 * nsys,), 0.5, dtype=torch.float32, device=dev)
    acc = torch.empty((2 * nsys, 3), dtype=torch.float32, device=dev)
    ctx = nb.NBody(2 * nsys, max_systems=nsys)
    ctx.build_tree_batched(x, m, torch.arange(0, 2 * nsys + 1, 2, device=dev))
    ctx.walk_groups(0.6, 8)
    ctx.forces(0.1, acc)
    ctx.close()
    d = pos.reshape(nsys, 2, 3)[:, ::-1].reshape(-1, 3) - pos
    want = 0.5 * d / ((d * d).sum(1) + 0.01)[:, None] ** 1.5
    # rsqrt to 1.3e-7, cubed, and a few roundings of 6e-8: below 1e-6
    assert np.abs(acc.cpu().numpy() - want).max() <= 1e-6 * np.abs(want).max()


@pytest.mark.parametrize("bad", [[0, 400, 900], [100, 500, 1000], [500, 1500, 1000],
                                 [0, 600, 500, 1000], [0, 500, 500, 1000], [0, 900, 800],
                                 [-5, 500, 1000], [300, 100, 1000], [900, 50, 100],
                                 [0, 2000, 3000]])
def test_offsets_that_are_no_partition_are_refused(bad):
    """Invalid argument, whatever an earlier batch left in the context, and the
    next batch is sorted as ever."""
    import paper_0909_0541_gb300 as nb
    n = 1000
    dev = torch.device("cuda")
    x = torch.from_numpy(nbsynth.uniform_cube(n, 3).pos).to(dev)
    m = torch.full((n,), 1.0 / n, dtype=torch.float32, device=dev)
    good = torch.tensor([0, 100, 200, 300, 400, 1000], device=dev)
    ctx = nb.NBody(n, max_systems=5)
    ctx.build_tree_batched(x, m, good)
    ref = ctx.copy_tree()
    with pytest.raises(nb.NBError) as e:
        ctx.build_tree_batched(x, m, torch.tensor(bad, device=dev))
    assert e.value.code == -1
    ctx.build_tree_batched(x, m, good)
    t = ctx.copy_tree()
    assert all(np.array_equal(ref[k], t[k]) for k in ("keys", "perm", "first", "count", "com"))
    ctx.close()

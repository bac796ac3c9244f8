"""Sizes where the launches and the force work items change: one block builds
the topology and the groups up to 4096 particles (1024 threads, 1, 2 or 4 keys
each), items hold 8
targets up to 8192 particles, 16 up to 32,768, then 32.  Trees, groups and
lists must equal the oracle's bit for bit on both sides of every line, forces
meet the tolerances of the parity tests, and the fused and overlapped passes
sum the same items in the same order (the same bits).
"""
import numpy as np
import pytest

import nbsynth
from tests.gpu_common import gpu_run
from tests.test_gpu_parity import assert_lists_equal, assert_tree_equal, clump_set

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)


@pytest.mark.parametrize("order", ["morton", "hilbert"])
@pytest.mark.parametrize("n,n_crit", [(1, 1), (2, 1), (33, 8), (1023, 32), (1024, 1), (1025, 64),
                                      (2048, 17), (2049, 64), (3000, 8192), (4095, 17), (4096, 64),
                                      (4097, 64), (8193, 64)])
def test_tree_groups_lists(oracle_lib, n, n_crit, order):
    ps = nbsynth.halo_mix(n, 60 + n, n_halos=5) if n > 100 else nbsynth.plummer(n, 60 + n)
    g = gpu_run(ps.pos, ps.mass, theta=0.7, n_crit=n_crit, eps=1e-3, key_order=order)
    T = oracle_lib.Tree(ps.pos, ps.mass, order=order)
    assert_tree_equal(g, T)
    if n_crit > 1 or n < 100:
        assert_lists_equal(g, T, 0.7, n_crit)


@pytest.mark.parametrize("n", [1000, 2000, 4096])
def test_deep_chains_and_coincident_points(oracle_lib, n):
    """Pairs 1e-6 apart and coincident points: cells down to the last level,
    several nodes per particle."""
    rng = np.random.default_rng(n)
    pos, mass = clump_set(n, n)
    k = n // 3
    pos[:k] = pos[k:2 * k] + 1e-6 * rng.normal(size=(k, 3))
    pos[5:25] = pos[4]
    g = gpu_run(pos, mass, theta=0.6, n_crit=16, eps=1e-3)
    T = oracle_lib.Tree(pos, mass)
    assert_tree_equal(g, T)
    assert_lists_equal(g, T, 0.6, 16)


@pytest.mark.parametrize("n", [8192, 8193, 32768, 32769])
def test_items_on_both_sides_of_a_line(oracle_lib, n):
    import paper_0909_0541_gb300 as nb
    ps = nbsynth.halo_mix(n, 70 + n, n_halos=12)
    theta, n_crit, eps = 0.7, 200, 1e-3
    T = oracle_lib.Tree(ps.pos, ps.mass)
    a, p, _, _, am = T.forces(n_crit, theta, eps, with_amag=True, coords32=True)
    dev = torch.device("cuda")
    x, m = torch.from_numpy(ps.pos).to(dev), torch.from_numpy(ps.mass).to(dev)
    for precision, tol in (("fp32", 1e-5), ("fp32_comp", 1e-6)):
        g = gpu_run(ps.pos, ps.mass, theta=theta, n_crit=n_crit, eps=eps, precision=precision,
                    lists=False)
        d = np.linalg.norm(g["acc"].astype(np.float64) - a, axis=1)
        assert np.all(d <= tol * am)
        assert np.all(np.abs(g["pot"] - p) <= tol * np.abs(p))
        ctx = g["ctx"]
        for other in (ctx.walk_forces, ctx.forces_fused):
            acc = torch.empty((n, 3), dtype=torch.float32, device=dev)
            pot = torch.empty(n, dtype=torch.float32, device=dev)
            other(theta, n_crit, eps, acc, pot, precision)
            assert np.array_equal(acc.cpu().numpy(), g["acc"])
            assert np.array_equal(pot.cpu().numpy(), g["pot"])
        ctx.close()


@pytest.mark.parametrize("n", [3000, 20000])
def test_autotuner_times_one_width_where_there_is_one(n):
    """Up to 1.5M particles both item widths form the same items: one timing,
    reported for both, and the wider one kept for later builds."""
    import paper_0909_0541_gb300 as nb
    ps = nbsynth.plummer(n, 9)
    dev = torch.device("cuda")
    ctx = nb.NBody(n)
    pick, table = ctx.autotune(torch.from_numpy(ps.pos).to(dev), torch.from_numpy(ps.mass).to(dev),
                               1e-3, 0.7, n_crits=(16, 64, 256), reps=2)
    ctx.close()
    assert pick["rows"] == 2
    for (crit, rows, tile, block), ms in table.items():
        assert ms > 0 and ms == table[(crit, 3 - rows, tile, block)]

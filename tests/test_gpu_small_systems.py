"""Sizes where the force work items change: they hold 8 targets up to 8192
particles, 16 up to 32,768, then 32.  On both sides of a line forces meet the
tolerances of the parity tests, and the fused and overlapped passes sum the
same items in the same order (the same bits).
"""
import numpy as np
import pytest

import nbsynth
from tests.gpu_common import gpu_run

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)


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

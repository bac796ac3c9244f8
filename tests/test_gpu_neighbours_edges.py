"""The neighbour search at the edges of its FP32 pair test, of its work items
and of its run sort, against the oracle's brute-force definition.

The sets are decided by the FP64 definition whatever the FP32 band leaves
open, so the CSR arrays must be equal element for element: on lattices whose
spacing is the radius (every pair of interest inside the band), far from the
origin (FP32 coordinates off by more than the band's first term), at scales
whose squares leave FP32's range (every pair left to FP64), for groups at the
64-member edge of a work item, and for runs at the edges of the register sort.
"""
import numpy as np
import pytest

import nbsynth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)


def gpu_neigh(pos, h, n_crit, offsets=None):
    import paper_0909_0541_gb300 as nb
    dev = torch.device("cuda")
    n = len(pos)
    p = torch.from_numpy(np.ascontiguousarray(pos, np.float64)).to(dev)
    m = torch.full((n,), 1.0 / n, dtype=torch.float32, device=dev)
    ctx = nb.NBody(n, max_systems=1 if offsets is None else len(offsets) - 1)
    if offsets is None:
        ctx.build_tree(p, m)
    else:
        ctx.build_tree_batched(p, m, torch.tensor(offsets, dtype=torch.int64, device=dev))
    off, idx = ctx.neighbours(h, n_crit)
    ctx.close()
    return off.cpu().numpy(), idx.cpu().numpy().astype(np.int64)


@pytest.mark.parametrize("scale", [1.0, 1e-12, 1e-18, 1e18])
@pytest.mark.parametrize("shift", [0.0, 1e3, 1e6])
def test_band_decides_as_the_definition(oracle_lib, scale, shift):
    g = np.arange(9) * 0.125
    lat = np.stack(np.meshgrid(g, g, g, indexing="ij"), -1).reshape(-1, 3)
    cube = nbsynth.uniform_cube(1500, 31).pos
    for pos, hs in ((lat, (0.125, 0.25)), (cube, (0.07, 0.2))):
        x = (pos + shift) * scale
        for h in hs:
            off, idx = gpu_neigh(x, h * scale, 64)
            ob, ib = oracle_lib.neighbours_brute(x, h * scale)
            assert np.array_equal(off, ob) and np.array_equal(idx, ib), (scale, shift, h)


@pytest.mark.parametrize("n,n_crit", [(63, 64), (64, 64), (65, 65), (97, 128), (129, 256),
                                      (257, 300), (1100, 2000), (1000, 63)])
def test_work_item_edges(oracle_lib, n, n_crit):
    pos = nbsynth.plummer(n, 60 + n).pos
    for h in (0.1, 1.0):
        off, idx = gpu_neigh(pos, h, n_crit)
        ob, ib = oracle_lib.neighbours_brute(pos, h)
        assert np.array_equal(off, ob) and np.array_equal(idx, ib), (n, n_crit, h)


@pytest.mark.parametrize("n", [2, 32, 33, 34, 65, 66, 129, 130, 257, 258, 600])
def test_run_sort_edges(n):
    """Everyone within reach: n - 1 neighbours each, in ascending order."""
    pos = nbsynth.uniform_cube(n, 80 + n).pos
    off, idx = gpu_neigh(pos, 10.0, 64)
    assert np.array_equal(off, np.arange(n + 1) * (n - 1))
    i = np.arange(n)
    want = np.concatenate([np.delete(i, k) for k in i])
    assert np.array_equal(idx, want)


def test_systems_of_unlike_scale(oracle_lib):
    """A batch searches each system alone, a small one beside a large one."""
    a = nbsynth.uniform_cube(700, 91).pos
    b = nbsynth.uniform_cube(500, 92).pos * 1e-3 + 3.0
    off, idx = gpu_neigh(np.concatenate([a, b]), 2e-4, 32, [0, 700, 1200])
    oa, ia = oracle_lib.neighbours_brute(a, 2e-4)
    ob, ib = oracle_lib.neighbours_brute(b, 2e-4)
    assert np.array_equal(off, np.concatenate([oa, oa[-1] + ob[1:]]))
    assert np.array_equal(idx, np.concatenate([ia, ib + 700]))

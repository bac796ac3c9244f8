"""Neighbour searches on one context, whose room for the answer comes from the
last search's: the CSR arrays equal the definition whether the room fits, is too
small, too large or cannot be had.
"""
import numpy as np
import pytest

import nbsynth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)


def _search(ctx, pos, h, oracle_lib):
    off, idx = ctx.neighbours(h, 64)
    ob, ib = oracle_lib.neighbours_brute(pos, h)
    assert np.array_equal(off.cpu().numpy(), ob)
    assert np.array_equal(idx.cpu().numpy().astype(np.int64), ib)
    # the table is not much larger than the answer it holds
    assert idx.untyped_storage().nbytes() <= 4 * (idx.numel() * 4 / 3 + 1)
    return off, idx


def test_searches_on_one_context(oracle_lib):
    """Growing, shrinking and empty searches, and searches after builds of
    fewer and of more particles."""
    import paper_0909_0541_gb300 as nb
    dev = torch.device("cuda")
    ctx = nb.NBody(6000)
    kept = []
    for n in (3000, 500, 6000):
        ps = nbsynth.uniform_cube(n, 20 + n)
        x, m = torch.from_numpy(ps.pos).to(dev), torch.from_numpy(ps.mass).to(dev)
        ctx.build_tree(x, m)
        for h in (0.05, 0.3, 0.31, 0.3, 0.05, 0.0, 1e-9, 0.0, 0.1, 0.2):
            kept.append(_search(ctx, ps.pos, h, oracle_lib) + (ps.pos, h))
    ctx.close()
    for off, idx, pos, h in kept[::7]:      # earlier answers stay what they were
        ob, ib = oracle_lib.neighbours_brute(pos, h)
        assert np.array_equal(idx.cpu().numpy().astype(np.int64), ib)


def test_search_when_the_last_search_was_too_large_to_repeat(oracle_lib):
    """Room for the last search's count that cannot be had (here 16 TB): the
    search counts first, as a context's first one does."""
    import paper_0909_0541_gb300 as nb
    ps = nbsynth.uniform_cube(800, 33)
    ctx = nb.NBody(800)
    ctx.build_tree(torch.from_numpy(ps.pos).cuda(), torch.from_numpy(ps.mass).cuda())
    _search(ctx, ps.pos, 0.2, oracle_lib)
    ctx._neigh_cap = 1 << 42
    _search(ctx, ps.pos, 0.1, oracle_lib)
    _search(ctx, ps.pos, 0.1, oracle_lib)
    ctx.close()

"""gs_bin_tiles on both sides of the choice between counting and the pair sort by the
number of primitives, one tile or two each.  The reference is numpy's stable sort."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [(1 << 20), (1 << 20) + 1])
@pytest.mark.parametrize("tx,ty", [(100, 90), (91, 99), (139, 100)])
def test_lists_of_large_scenes(n, tx, ty):
    import torch

    import paper_2606_21791_gb300 as P
    P.build()
    from paper_2606_21791_gb300 import gs as G
    G.load_library()
    rng = np.random.default_rng(n + tx)
    depth = np.round(rng.uniform(0.5, 40.0, n), 2).astype(np.float32)   # many ties
    x, y = rng.integers(0, tx, n), rng.integers(0, ty, n)
    w = rng.integers(0, 3, n)   # nothing, one tile, two
    rects = np.stack([x, y, np.minimum(x + w, tx), y + 1], axis=1).astype(np.int32)
    wide = np.minimum(x + w, tx) - x
    prim = np.repeat(np.arange(n), wide)
    tile = (y * tx + x)[prim] + np.concatenate([[0], (prim[1:] == prim[:-1]).astype(int)])
    order = np.lexsort((prim, depth[prim], tile))
    off = torch.zeros(tx * ty + 1, dtype=torch.int32, device="cuda")
    ids = torch.zeros(len(prim), dtype=torch.int32, device="cuda")
    assert G.gs_bin_tiles(torch.from_numpy(depth).cuda(), torch.from_numpy(rects).cuda(), n, tx, ty, off, ids,
                          len(prim)) == len(prim)
    assert np.array_equal(ids.cpu().numpy(), prim[order])
    assert np.array_equal(off.cpu().numpy(), np.concatenate([[0], np.cumsum(np.bincount(tile, minlength=tx * ty))]))


@pytest.mark.parametrize("cap", [(1 << 22), (1 << 22) + 1])
def test_pair_sort_around_the_block_sizes(cap):
    """Pair capacities on both sides of a radix pass's change of items per thread: the
    same lists."""
    import torch

    import paper_2606_21791_gb300 as P
    P.build()
    from paper_2606_21791_gb300 import gs as G
    G.load_library()
    n, tx, ty = 50_000, 160, 122
    rng = np.random.default_rng(7)
    depth = rng.uniform(0.5, 40.0, n).astype(np.float32)
    x, y = rng.integers(0, tx - 8, n), rng.integers(0, ty, n)
    rects = np.stack([x, y, x + 8, y + 1], axis=1).astype(np.int32)
    tile = ((y * tx + x)[:, None] + np.arange(8)).reshape(-1)
    prim = np.repeat(np.arange(n), 8)
    order = np.lexsort((prim, depth[prim], tile))
    off = torch.zeros(tx * ty + 1, dtype=torch.int32, device="cuda")
    ids = torch.zeros(cap, dtype=torch.int32, device="cuda")
    assert G.gs_bin_tiles(torch.from_numpy(depth).cuda(), torch.from_numpy(rects).cuda(), n, tx, ty, off, ids,
                          cap) == 8 * n
    assert np.array_equal(ids.cpu().numpy()[:8 * n], prim[order])

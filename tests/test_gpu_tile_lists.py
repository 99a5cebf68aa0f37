"""gs_bin_tiles where its paths split: primitive counts around the one-block order
and the radix passes' block sizes, tile grids around the limit of the counting
lists, primitives that cover nothing, one tile or the whole grid, depth ties.
The reference is numpy's stable sort by (tile, depth, primitive)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def G():
    import paper_2606_21791_gb300 as P
    P.build()
    from paper_2606_21791_gb300 import gs
    gs.load_library()
    return gs


def _inputs(n, tx, ty, seed, big):
    rng = np.random.default_rng(seed)
    depth = np.round(rng.uniform(0.5, 40.0, n), 1).astype(np.float32)      # many ties
    x0, y0 = rng.integers(-2, tx, n), rng.integers(-2, ty, n)
    r = np.stack([x0, y0, x0 + rng.integers(-1, 4, n), y0 + rng.integers(-1, 4, n)], axis=1).astype(np.int32)
    k = rng.choice(n, min(big, n), replace=False)
    r[k] = [-5, -5, tx + 9, ty + 9]                                        # the whole grid
    return depth, r


def _reference(depth, r, tx, ty):
    x0, y0 = np.clip(r[:, 0], 0, tx), np.clip(r[:, 1], 0, ty)
    x1, y1 = np.clip(r[:, 2], 0, tx), np.clip(r[:, 3], 0, ty)
    tiles, prims = [], []
    for i in np.flatnonzero((x1 > x0) & (y1 > y0)):
        t = (np.arange(y0[i], y1[i])[:, None] * tx + np.arange(x0[i], x1[i])).reshape(-1)
        tiles.append(t)
        prims.append(np.full(len(t), i))
    if not tiles:
        return np.zeros(tx * ty + 1, np.uint32), np.zeros(0, np.uint32)
    tiles, prims = np.concatenate(tiles), np.concatenate(prims)
    order = np.lexsort((prims, depth[prims], tiles))
    off = np.concatenate([[0], np.cumsum(np.bincount(tiles, minlength=tx * ty))])
    return off.astype(np.uint32), prims[order].astype(np.uint32)


@pytest.mark.parametrize("tx,ty", [(1, 1), (7, 3), (100, 65), (139, 100), (140, 100), (251, 3)])
@pytest.mark.parametrize("n,big", [(1, 0), (33, 2), (8191, 3), (8192, 0), (8193, 3), (20000, 1)])
def test_bin_tiles(G, n, big, tx, ty):
    import torch
    depth, r = _inputs(n, tx, ty, n * 31 + tx, big)
    off_ref, ids_ref = _reference(depth, r, tx, ty)
    d, rr = torch.from_numpy(depth).cuda(), torch.from_numpy(r).cuda()
    off = torch.zeros(tx * ty + 1, dtype=torch.int32, device="cuda")
    for cap in (max(len(ids_ref), 1), 3 * len(ids_ref) + 1000):
        ids = torch.zeros(cap, dtype=torch.int32, device="cuda")
        total = G.gs_bin_tiles(d, rr, n, tx, ty, off, ids, cap)
        assert total == len(ids_ref)
        assert np.array_equal(off.cpu().numpy().view(np.uint32), off_ref)
        assert np.array_equal(ids.cpu().numpy().view(np.uint32)[:total], ids_ref)
    if len(ids_ref) > 1:
        with pytest.raises(G.GsError) as e:
            G.gs_bin_tiles(d, rr, n, tx, ty, off, ids, len(ids_ref) - 1)
        assert e.value.status == G.GS_ERR_CAPACITY


@pytest.mark.parametrize("n", [520_000, 530_000])
def test_bin_tiles_around_the_block_sizes(G, n):
    """Around 2^19 primitives, where a radix pass changes its items per thread."""
    import torch
    depth, r = _inputs(n, 40, 30, n, 2)
    r[:, 2:] = np.minimum(r[:, 2:], r[:, :2] + 1)   # one tile each: a quick reference
    off_ref, ids_ref = _reference(depth, r, 40, 30)
    off = torch.zeros(1201, dtype=torch.int32, device="cuda")
    ids = torch.zeros(len(ids_ref), dtype=torch.int32, device="cuda")
    assert G.gs_bin_tiles(torch.from_numpy(depth).cuda(), torch.from_numpy(r).cuda(), n, 40, 30, off, ids,
                          len(ids_ref)) == len(ids_ref)
    assert np.array_equal(off.cpu().numpy().view(np.uint32), off_ref)
    assert np.array_equal(ids.cpu().numpy().view(np.uint32), ids_ref)

"""The dirty-tile engine where its paths split: pixel blend lists cut short,
large batches in tile order against small ones, needle-shaped primitives (whose
determinants the plan's margins lose), other tile shapes in large batches.  The
reference is the full re-render of each variant, bit for bit."""
import numpy as np
import pytest

from paper_2606_21791_gb300 import synth as S

pytestmark = pytest.mark.gpu
FIELDS = ("sse", "maxabs", "footprint", "nonfinite", "clamps")


@pytest.fixture(scope="module")
def G():
    import paper_2606_21791_gb300 as P
    P.build()
    from paper_2606_21791_gb300 import gs
    gs.load_library()
    return gs


def _run(G, h, flips, K, full=False, guard=-1):
    import torch
    out = G.device_bytes(len(flips) * K * 24)
    fn = G.gs_inject_and_render_full if full else G.gs_inject_and_render
    fn(h, G.to_device(flips), len(flips), 1, guard, S.GUARD_WORDS_DEFAULT, out)
    torch.cuda.synchronize()
    return G.from_device(out, G.RESULT_DTYPE).reshape(len(flips), K)


def _same(a, b):
    for f in FIELDS:
        assert np.array_equal(a[f], b[f]), f


def test_cut_lists(G):
    """400 large, barely visible primitives over every pixel of a 1600x1040 view:
    more list entries than are kept, so the walks end in the tile's own list."""
    n = 400
    v = S.scene_values(n, 0, S.SEED_BASE + 300, layout="cube")
    rng = np.random.default_rng(300)
    v[0:2] = rng.uniform(-1, 1, size=(2, n))
    v[3:6] = rng.uniform(2.0, 2.5, size=(3, n))     # scales of 7 to 12 at distance 15: the whole view
    v[10] = rng.uniform(-4.6, -4.2, size=n)          # opacities of 0.010 to 0.015: no pixel stops early
    sc = S.Scene(planes=S.encode(v, S.FP32), fmt=S.FP32, sh_degree=0)
    cams = S.ring_cameras(1, 1600, 1040)
    prim = np.array([3, 7, 120, 250, 399, 10, 77, 301], dtype=np.uint32)
    word = np.array([10, 10, 11, 10, 2, 5, 12, 4])
    bit = np.array([30, 31, 22, 23, 22, 23, 31, 31])
    flips = S.flips_at(prim, word, bit)
    h = G.gs_load_scene(sc.planes, sc.n, 0, S.FP32)
    try:
        G.gs_set_views(h, cams)
        a, b = _run(G, h, flips, 1), _run(G, h, flips, 1, full=True)
        _same(a, b)
        assert (a["sse"] > 0).sum() >= 6
    finally:
        G.gs_free_scene(h)


@pytest.mark.parametrize("K,W,H,tile", [(1, 320, 240, (16, 16)), (3, 250, 131, (16, 16)), (2, 320, 240, (8, 8)),
                                        (1, 333, 200, (32, 8))])
def test_large_batches_equal_small_ones(G, K, W, H, tile):
    """One batch of all upsets (tile order) against batches of 100 (as planned), and
    a sample of full re-renders."""
    sc = S.make_scene(20000, 1, S.FP32, S.SEED_BASE + 310, layout="clusters")
    flips = S.flips_stratified(20000, sc.n, sc.nwords, S.FP32, 311)
    h = G.gs_load_scene(sc.planes, sc.n, 1, S.FP32)
    try:
        G.gs_set_tile(h, *tile)
        G.gs_set_views(h, S.ring_cameras(K, W, H))
        a = _run(G, h, flips, K)
        G.gs_set_batch(h, 100)
        _same(a[::7], _run(G, h, flips[::7], K))
        _same(a[::199], _run(G, h, flips[::199], K, full=True))
    finally:
        G.gs_free_scene(h)


@pytest.mark.parametrize("seed", [0, 1])
@pytest.mark.parametrize("n,degree", [(3000, 0), (60000, 0)])
def test_needles(G, n, degree, seed):
    """Log-scale sign and exponent upsets: primitives that explode along one axis,
    crossing the view as needles and bands."""
    sc = S.make_scene(n, degree, S.FP32, S.SEED_BASE + 320 + seed, layout="clusters")
    rng = np.random.default_rng(321 + seed)
    cnt = 160
    flips = S.flips_at(rng.integers(0, n, cnt).astype(np.uint32), rng.integers(3, 6, cnt), rng.integers(24, 32, cnt))
    K = 2
    h = G.gs_load_scene(sc.planes, sc.n, degree, S.FP32)
    try:
        G.gs_set_views(h, S.ring_cameras(K, 640, 433))
        a = _run(G, h, flips, K)
        _same(a, _run(G, h, flips, K, full=True))
        assert (a["footprint"] > 0).sum() > cnt // 4
    finally:
        G.gs_free_scene(h)


def test_changes_before_and_behind_the_stop(G):
    """Opacity and depth upsets of single primitives in deep lists: the removed and the
    inserted entry anywhere in a pixel's list, apart, together, at its end."""
    sc = S.make_scene(40000, 0, S.FP32, S.SEED_BASE + 330, layout="clusters")
    rng = np.random.default_rng(331)
    cnt = 600
    word = rng.choice([0, 1, 2, 10], cnt)
    bit = np.where(word == 10, rng.integers(20, 32, cnt), rng.integers(14, 24, cnt))
    flips = S.flips_at(rng.integers(0, sc.n, cnt).astype(np.uint32), word, bit)
    h = G.gs_load_scene(sc.planes, sc.n, 0, S.FP32)
    try:
        G.gs_set_views(h, S.ring_cameras(1, 256, 256))
        _same(_run(G, h, flips, 1), _run(G, h, flips, 1, full=True))
    finally:
        G.gs_free_scene(h)

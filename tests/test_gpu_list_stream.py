"""Clean views against the other blends at the edges of their batches: the clean
passes stream a tile's list in batches of one entry per thread and drop entries by
their ellipses, gs_render stages it and drops by ellipses, the full re-renders
stage it and drop by boxes.  All three have to take the same entries: bit for bit."""
import numpy as np
import pytest

from paper_2606_21791_gb300 import synth as S

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def G():
    import paper_2606_21791_gb300 as P
    P.build()
    from paper_2606_21791_gb300 import gs
    gs.load_library()
    return gs


def _scene(n, seed):
    """n - 1 slanted, flat, see-through primitives over the middle of the view and
    one behind the camera."""
    v = S.scene_values(n, 0, seed, layout="cube")
    rng = np.random.default_rng(seed)
    v[0:3] = rng.uniform([[-6.0], [-4.0], [-1.5]], [[6.0], [4.0], [1.5]], size=(3, n))
    v[3:6] = rng.uniform([[-4.5], [-4.5], [-0.5]], [[-2.5], [-2.5], [0.8]], size=(3, n))
    v[10] = rng.uniform(-4.0, -1.0, size=n)
    v[0:3, n - 1] = (0.0, 0.0, 20.0)   # the first camera of the ring stands at (0, 0, 15) and looks at 0
    return S.Scene(planes=S.encode(v, S.FP32), fmt=S.FP32, sh_degree=0), S.ring_cameras(1, 61, 43)


@pytest.mark.parametrize("tile", [(16, 16), (8, 8), (32, 8)])
@pytest.mark.parametrize("n", [2, 32, 33, 64, 65, 128, 129, 130, 256, 257, 258, 385, 1000])
def test_same_entries(G, n, tile):
    import torch
    sc, cam = _scene(n, S.SEED_BASE + 400 + n)
    flips = S.flips_at(np.array([n - 1], dtype=np.uint32), np.array([10]), np.array([0]))   # changes nothing seen
    h = G.gs_load_scene(sc.planes, sc.n, 0, S.FP32)
    try:
        G.gs_set_tile(h, *tile)
        G.gs_set_views(h, cam)
        out = G.device_bytes(24)
        G.gs_inject_and_render_full(h, G.to_device(flips), 1, 1, -1, S.GUARD_WORDS_DEFAULT, out)
        torch.cuda.synchronize()
        r = G.from_device(out, G.RESULT_DTYPE)[0]
        assert r["sse"] == 0 and r["maxabs"] == 0 and r["footprint"] == 0 and r["nonfinite"] == 0
        a = torch.empty(1, 43, 61, 3, device="cuda")
        b = torch.empty_like(a)
        G.gs_clean_image(h, 0, a)
        G.gs_render(h, cam, b)
        torch.cuda.synchronize()
        assert torch.equal(a.view(torch.int32), b.view(torch.int32))
        assert n < 100 or (a < 0.99).float().mean() > 0.2   # the lists are there
    finally:
        G.gs_free_scene(h)

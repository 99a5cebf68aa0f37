"""Dense views: nearly every entry of an 8x8 block is taken at every pixel, so the view
keeps block lists in place of its pixels' blend lists.  The reference is the full
re-render of each variant, bit for bit; a far camera on the same scene gives a view with
blend lists beside a dense one."""
import numpy as np
import pytest

from paper_2606_21791_gb300 import synth as S

pytestmark = pytest.mark.gpu
W, H, N = 640, 433, 4000


@pytest.fixture(scope="module")
def G():
    import paper_2606_21791_gb300 as P
    P.build()
    from paper_2606_21791_gb300 import gs
    gs.load_library()
    return gs


def _scene(nan=False):
    """Primitives of 0.4 to 0.7 at distance 15: standard deviations of 9 to 16 pixels."""
    v = S.scene_values(N, 0, S.SEED_BASE + 430, layout="cube")
    rng = np.random.default_rng(430)
    v[0:2] = rng.uniform(-4, 4, size=(2, N))
    v[3:6] = rng.uniform(-1.0, -0.4, size=(3, N))
    v[10] = rng.uniform(-2.0, 2.0, size=N)
    if nan:   # a few clean primitives of NaN colour or opacity
        v[11, :3] = np.nan
        v[10, 3:5] = np.nan
    return S.Scene(planes=S.encode(v, S.FP32), fmt=S.FP32, sh_degree=0)


def _cams(far):
    near = S.ring_cameras(2, W, H)
    if not far:
        return near
    return np.concatenate([near[:1], S.ring_cameras(1, W, H, distance=400.0), near[1:]])


def _flips(cnt, seed):
    rng = np.random.default_rng(seed)
    word, bit = rng.integers(0, 14, cnt), rng.integers(12, 32, cnt)
    return S.flips_at(rng.integers(0, N, cnt).astype(np.uint32), word, bit)


def _run(G, h, flips, K, full=False, guard=-1):
    import torch
    out = G.device_bytes(len(flips) * K * 24)
    fn = G.gs_inject_and_render_full if full else G.gs_inject_and_render
    fn(h, G.to_device(flips), len(flips), 1, guard, S.GUARD_WORDS_DEFAULT, out)
    torch.cuda.synchronize()
    return G.from_device(out, G.RESULT_DTYPE).reshape(len(flips), K)


@pytest.mark.parametrize("tile", [(16, 16), (8, 8), (32, 8)])
@pytest.mark.parametrize("far", [False, True])
def test_records_equal_full_rerenders(G, far, tile):
    import torch
    sc, cams, flips = _scene(), _cams(far), _flips(260, 431)
    h = G.gs_load_scene(sc.planes, N, 0, S.FP32)
    try:
        G.gs_set_tile(h, *tile)
        free = torch.cuda.mem_get_info()[0]
        G.gs_set_views(h, cams)
        # blend lists of a near view alone would take more (60 entries of 24 B a pixel)
        assert free - torch.cuda.mem_get_info()[0] < 300 << 20
        a = _run(G, h, flips, len(cams))
        assert (a["sse"] > 0).sum() > 100
        full = _run(G, h, flips, len(cams), full=True)
        assert a.tobytes() == full.tobytes()
        G.gs_set_batch(h, 30)
        assert a.tobytes() == _run(G, h, flips, len(cams)).tobytes()
        assert _run(G, h, flips[::9], len(cams), guard=0).tobytes() == _run(G, h, flips[::9], len(cams), full=True,
                                                                        guard=0).tobytes()
    finally:
        G.gs_free_scene(h)


def test_nan_primitives(G):
    sc, cams, flips = _scene(nan=True), _cams(True), _flips(120, 432)
    flips["prim"][:40] = np.arange(40) % 6   # the NaN primitives themselves
    h = G.gs_load_scene(sc.planes, N, 0, S.FP32)
    try:
        G.gs_set_views(h, cams)
        a = _run(G, h, flips, len(cams))
        assert (a["nonfinite"] > 0).any()
        assert a.tobytes() == _run(G, h, flips, len(cams), full=True).tobytes()
    finally:
        G.gs_free_scene(h)


def test_ssim_and_regions(G):
    """SSIM and contamination masks of a dense view and of one with lists beside it."""
    import torch
    sc, cams, flips = _scene(), _cams(True), _flips(48, 433)
    K, B = len(cams), 48
    h = G.gs_load_scene(sc.planes, N, 0, S.FP32)
    try:
        G.gs_set_views(h, cams)
        out, reg = G.device_bytes(B * K * 24), torch.zeros(B * K, 2, dtype=torch.int64, device="cuda")
        ss = torch.zeros(B * K, dtype=torch.float64, device="cuda")
        G.gs_inject_and_render_ex(h, G.to_device(flips), B, -1, 0, out, reg, ss)
        torch.cuda.synchronize()
        reg, ss = reg.cpu().numpy().reshape(B, K, 2), ss.cpu().numpy().reshape(B, K)
        clean = torch.empty(K, H, W, 3, device="cuda")
        for k in range(K):
            G.gs_clean_image(h, k, clean[k])
        img, one = torch.empty_like(clean), torch.zeros(K, dtype=torch.float64, device="cuda")
        y, x = np.mgrid[0:H, 0:W]
        cell = (8 * y // H) * 8 + 8 * x // W
        for i in range(0, B, 3):
            f = G.to_device(flips[i:i + 1])
            G.gs_apply_flips(h, f, 1)
            G.gs_render(h, cams, img)
            G.gs_apply_flips(h, f, 1)   # XOR back
            G.gs_ssim(img, clean, H, W, K, one)
            torch.cuda.synchronize()
            assert np.array_equal(one.cpu().numpy(), ss[i])
            d = (torch.nan_to_num(img, nan=0.0).clamp(0, 1) - clean.clamp(0, 1)).abs().amax(dim=3).cpu().numpy()
            for k in range(K):
                want = 0
                for c in np.unique(cell[d[k] > np.float32(1.0 / 255.0)]):
                    want |= 1 << int(c)
                assert int(reg[i, k, 0]) & (2**64 - 1) == want
    finally:
        G.gs_free_scene(h)

"""gs_compare and gs_ssim at the sizes and alignments where their loads and tiles
split: images of one pixel up to several tiles, pixel counts with every remainder
of four, images that start off a 16-byte boundary, several pairs in one call."""
import numpy as np
import pytest

import oracle as O

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def G():
    import paper_2606_21791_gb300 as P
    P.build()
    from paper_2606_21791_gb300 import gs
    gs.load_library()
    return gs


def _pairs(seed, K, H, W):
    rng = np.random.default_rng(seed)
    a = rng.uniform(-0.2, 1.2, size=(K, H, W, 3)).astype(np.float32)
    b = a + (rng.normal(0, 0.02, size=a.shape) * (rng.uniform(size=a.shape) < 0.5)).astype(np.float32)
    a[0, H // 2, W // 2, 1] = np.nan
    a[K - 1, 0, 0, 2] = -np.inf
    return a, b


def _device(x, shift):
    """The array on the device, starting `shift` floats past an allocation."""
    import torch
    buf = torch.zeros(x.size + shift, dtype=torch.float32, device="cuda")
    buf[shift:] = torch.from_numpy(x.reshape(-1).copy()).cuda()
    return buf, buf.data_ptr() + 4 * shift


@pytest.mark.parametrize("shift", [0, 1, 2, 4])
@pytest.mark.parametrize("K,H,W", [(1, 1, 1), (2, 1, 3), (3, 5, 7), (2, 16, 16), (1, 33, 129), (5, 64, 97),
                                   (2, 401, 331)])
def test_compare_sizes_and_alignments(G, K, H, W, shift):
    import torch
    a, b = _pairs(K * 1000 + H + W, K, H, W)
    ka, pa = _device(a, shift)
    kb, pb = _device(b, 4)
    out = G.device_bytes(K * 24)
    G.gs_compare(pa, pb, H, W, K, out)
    torch.cuda.synchronize()
    r = G.from_device(out, G.RESULT_DTYPE)
    for k in range(K):
        o = O.compare(a[k], b[k])
        assert r[k]["footprint"] == o["footprint"] and r[k]["nonfinite"] == o["nonfinite"]
        assert r[k]["maxabs"] == o["maxabs"]
        # each pixel's squared error is rounded to 2^-39 and to fp32 (relative 2^-22 for its three terms)
        assert abs(r[k]["sse"] - o["sse"]) <= H * W * 2.0 ** -39 + 2.0 ** -21 * o["sse"]


@pytest.mark.parametrize("K,H,W", [(1, 10, 40), (2, 11, 11), (1, 12, 27), (3, 16, 16), (2, 17, 33), (1, 26, 21),
                                   (2, 53, 70)])
def test_ssim_sizes(G, K, H, W):
    import torch
    a, b = _pairs(K * 77 + H * W, K, H, W)
    da, db = torch.from_numpy(a).cuda(), torch.from_numpy(b).cuda()
    out = torch.zeros(K, dtype=torch.float64, device="cuda")
    G.gs_ssim(db, da, H, W, K, out)
    torch.cuda.synchronize()
    o = np.array([O.ssim(b[k], a[k]) for k in range(K)])
    assert np.abs(out.cpu().numpy() - o).max() < 5e-5   # the repository's SSIM tolerance
    G.gs_ssim(da, da, H, W, K, out)
    torch.cuda.synchronize()
    assert (out.cpu().numpy() == 1.0).all()

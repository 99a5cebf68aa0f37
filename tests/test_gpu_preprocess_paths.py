"""The bulk-copy preprocess (one or two stages, by format and SH degree) against the
per-thread one, which scenes of an odd size take: the same records, bit for bit."""
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


def _records(G, planes, n, degree, fmt, cam):
    import torch
    h = G.gs_load_scene(np.ascontiguousarray(planes), n, degree, fmt)
    try:
        out = torch.zeros(n * 64, dtype=torch.uint8, device="cuda")
        G.gs_preprocess(h, cam, out)
        torch.cuda.synchronize()
        return out.cpu().numpy().reshape(n, 64)
    finally:
        G.gs_free_scene(h)


@pytest.mark.parametrize("fmt,degree", [(S.FP32, 3), (S.FP32, 2), (S.FP32, 0), (S.FP16, 3), (S.BF16, 1)])
@pytest.mark.parametrize("n", [8, 120, 128, 136, 264, 3000, 450000])
def test_same_records(G, fmt, degree, n):
    if n > 3000 and degree < 2:
        pytest.skip("several tiles a block: the large stages")
    sc = S.make_scene(n + 1, degree, fmt, S.SEED_BASE + 500, layout="clusters")
    cam = S.ring_cameras(1, 640, 360)
    a = _records(G, sc.planes[:, :n], n, degree, fmt, cam)
    b = _records(G, sc.planes, n + 1, degree, fmt, cam)
    assert np.array_equal(a, b[:n])
    assert a.any()

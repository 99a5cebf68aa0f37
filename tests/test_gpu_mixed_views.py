"""Full re-renders over a set of views of different sizes, one listed by counting and
one by the pair sort, in both orders: single upsets against the dirty-tile engine,
many upsets a variant against each view alone."""
import numpy as np
import pytest

from paper_2606_21791_gb300 import synth as S

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("sizes", [((640, 483), (2592, 1944)), ((2592, 1944), (640, 483))])
def test_full_rerender_over_views_of_different_sizes(sizes):
    import torch

    import paper_2606_21791_gb300 as P
    P.build()
    from paper_2606_21791_gb300 import gs as G
    G.load_library()
    sc = S.make_scene(20000, 1, S.FP32, S.SEED_BASE + 400, layout="clusters")
    cams = np.concatenate([S.ring_cameras(2, *s)[i:i + 1] for i, s in enumerate(sizes)])
    single = S.flips_top_bits(12, sc.n, sc.nwords, 401)
    many = S.flips_multi(2 * 2000, sc.n, sc.nwords, S.FP32, 402)

    def run(fn, flips, B, per, K):
        out = G.device_bytes(B * K * 24)
        fn(h, G.to_device(flips), B, per, -1, 0, out)
        torch.cuda.synchronize()
        return G.from_device(out, G.RESULT_DTYPE).reshape(B, K)

    h = G.gs_load_scene(sc.planes, sc.n, 1, S.FP32)
    try:
        G.gs_set_views(h, cams)
        a = run(G.gs_inject_and_render_full, single, 12, 1, 2)
        assert a.tobytes() == run(G.gs_inject_and_render, single, 12, 1, 2).tobytes()
        b = run(G.gs_inject_and_render, many, 2, 2000, 2)
        assert (b["footprint"] > 0).all()
        for k in range(2):
            G.gs_set_views(h, cams[k:k + 1])
            assert run(G.gs_inject_and_render, many, 2, 2000, 1).tobytes() == np.ascontiguousarray(b[:, k]).tobytes()
    finally:
        G.gs_free_scene(h)

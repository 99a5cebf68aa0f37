"""Batches whose candidates are covered by exploded primitives (the blend's units hold
few of them), hardly reached (a block's share in one unit) and mixed, against batches
of a few variants and against full re-renders, bit for bit."""
import numpy as np
import pytest

from paper_2606_21791_gb300 import synth as S

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kind", ["covered", "light", "mixed"])
@pytest.mark.parametrize("tile", [(16, 16), (8, 8)])
def test_units(kind, tile):
    import torch

    import paper_2606_21791_gb300 as P
    P.build()
    from paper_2606_21791_gb300 import gs as G
    G.load_library()
    sc = S.make_scene(6000, 0, S.FP32, S.SEED_BASE + 420, layout="clusters")
    rng = np.random.default_rng(421)
    cnt = 900
    covered = {"covered": np.ones(cnt, bool), "light": np.zeros(cnt, bool), "mixed": np.arange(cnt) % 9 == 0}[kind]
    # a log-scale's sign bit or low exponent bits; its upper mantissa bits
    bit = np.where(covered, rng.choice([23, 24, 31], cnt), rng.integers(14, 20, cnt))
    flips = S.flips_at(rng.integers(0, sc.n, cnt).astype(np.uint32), rng.integers(3, 6, cnt), bit)
    K = 2

    def run(fn, f):
        out = G.device_bytes(len(f) * K * 24)
        fn(h, G.to_device(f), len(f), 1, -1, 0, out)
        torch.cuda.synchronize()
        return G.from_device(out, G.RESULT_DTYPE).reshape(len(f), K)

    h = G.gs_load_scene(sc.planes, sc.n, 0, S.FP32)
    try:
        G.gs_set_tile(h, *tile)
        G.gs_set_views(h, S.ring_cameras(K, 800, 633))
        a = run(G.gs_inject_and_render, flips)
        assert (a["sse"] > 0).sum() > cnt // 8
        G.gs_set_batch(h, 16)
        assert a.tobytes() == run(G.gs_inject_and_render, flips).tobytes()
        s = slice(0, cnt, 45)
        assert np.ascontiguousarray(a[s]).tobytes() == run(G.gs_inject_and_render_full, np.ascontiguousarray(flips[s])).tobytes()
    finally:
        G.gs_free_scene(h)

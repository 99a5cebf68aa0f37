"""Variants per warp of the injector: large batches, where a warp takes several
variants (8 at most, K each), against batches of 100, where it takes one."""
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


@pytest.mark.parametrize("K,B,guard", [(1, 40001, "prim"), (3, 20003, "none"), (5, 13001, "field"), (5, 5003, "ecc"),
                                       (11, 5901, "prim"), (16, 4090, "field")])
def test_groups_equal_single_variants(G, K, B, guard):
    import torch
    mode = {"none": G.GS_GUARD_OFF, "field": G.GS_GUARD_FIELD, "prim": G.GS_GUARD_PRIM, "ecc": G.GS_GUARD_ECC}[guard]
    sc = S.make_scene(6000, 1, S.FP16, S.SEED_BASE + 600 + K, layout="clusters")
    flips = S.flips_stratified(B, sc.n, sc.nwords, S.FP16, 601)
    h = G.gs_load_scene(sc.planes, sc.n, 1, S.FP16)
    try:
        if guard == "prim":
            G.gs_set_prim_box(h, sc.planes, sc.planes, sc.nwords)
        if guard == "field":
            G.gs_field_box(h, sc.nwords)
        G.gs_set_views(h, S.ring_cameras(K, 96, 80))

        def run(f):
            out = G.device_bytes(len(f) * K * 24)
            G.gs_inject_and_render(h, G.to_device(f), len(f), 1, mode, S.GUARD_WORDS_DEFAULT, out)
            torch.cuda.synchronize()
            return G.from_device(out, G.RESULT_DTYPE).reshape(len(f), K)

        a = run(flips)
        G.gs_set_batch(h, 100)
        b = run(flips)
        assert a.tobytes() == b.tobytes()
        assert (a["clamps"] > 0).any() == (guard in ("field", "prim"))
        assert guard == "prim" or (a["footprint"] > 0).any()
    finally:
        G.gs_free_scene(h)

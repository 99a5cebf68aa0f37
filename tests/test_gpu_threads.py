"""Renders and view set-ups of several threads at once, on scenes of different sizes,
grids and tile shapes: every launch keeps its own shared-memory size, so images and
records equal those of one thread, bit for bit."""
import threading

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


def _job(G, n, degree, W, H, tile, rounds, out, errors):
    import torch
    try:
        torch.cuda.set_device(0)
        st = torch.cuda.Stream()
        with torch.cuda.stream(st):
            sc = S.make_scene(n, degree, S.FP32, S.SEED_BASE + 700 + n, layout="clusters")
            flips = G.to_device(S.flips_stratified(40, n, sc.nwords, S.FP32, 701))
            h = G.gs_load_scene(sc.planes, n, degree, S.FP32)
            try:
                G.gs_set_tile(h, *tile, stream=st)
                cams = S.ring_cameras(2, W, H)
                img = torch.empty(2, H, W, 3, device="cuda")
                res = G.device_bytes(40 * 2 * 24)
                for _ in range(rounds):
                    G.gs_render(h, cams, img, stream=st)
                    G.gs_set_views(h, cams, stream=st)
                    G.gs_inject_and_render(h, flips, 40, 1, -1, S.GUARD_WORDS_DEFAULT, res, stream=st)
                    st.synchronize()
                    out.append((img.cpu().numpy().tobytes(), G.from_device(res, G.RESULT_DTYPE).tobytes()))
            finally:
                G.gs_free_scene(h)
    except Exception as e:   # noqa: BLE001 - reported by the test
        errors.append(e)


def test_threads_equal_one_thread(G):
    jobs = [(9001, 0, 320, 240, (16, 16)), (20003, 1, 1600, 1040, (16, 16)), (30000, 2, 800, 800, (8, 8)),
            (12000, 3, 640, 480, (32, 8))]
    want = []
    for j in jobs:
        out, err = [], []
        _job(G, *j, 1, out, err)
        assert not err, err
        want.append(out[0])
    outs, errors = [[] for _ in jobs], []
    threads = [threading.Thread(target=_job, args=(G, *j, 12, o, errors)) for j, o in zip(jobs, outs)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors
    for o, w in zip(outs, want):
        assert len(o) == 12 and all(x == w for x in o)

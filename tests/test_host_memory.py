"""The host side of libgs without a GPU: its own objects linked against a stand-in
for the CUDA runtime (fake_cudart.cpp), which maps device memory lazily, runs no
kernel, and checks the arrays that some of them are given."""
import ctypes as C
import glob
import os
import subprocess
import sys
import textwrap

import pytest

from paper_2606_21791_gb300 import buildlib

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="session")
def fake():
    """Path of the library linked against the stand-in."""
    buildlib.build()
    objs = [os.path.join(buildlib.BUILD, os.path.basename(s)[:-3] + ".o") for s in buildlib._sources()]
    if not all(os.path.exists(o) for o in objs):
        buildlib.build(force=True)
    include = os.path.join(os.path.dirname(os.path.dirname(buildlib.nvcc())), "include")
    lib = os.path.join(buildlib.BUILD, "libgs_fake.so")
    src = os.path.join(HERE, "fake_cudart.cpp")
    cmd = ["g++", "-O1", "-std=c++17", "-fPIC", "-fvisibility=hidden", "-I", include, "-shared", "-Wl,-Bsymbolic",
           "-Wl,--no-undefined", "-o", lib, src, *objs, "-lpthread"]
    r = subprocess.run(cmd, capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    return lib


PRELUDE = """
import ctypes as C
import numpy as np
from paper_2606_21791_gb300 import gs as G, synth as S
L = G.load_library({lib!r})
for f in ("fake_live", "fake_allocations"):
    getattr(L, f).restype = C.c_uint64
L.fake_report.restype = C.c_char_p
L.fake_limit.argtypes = [C.c_uint64]
L.fake_counts.argtypes = [C.c_uint64] * 3
ADDR = 1 << 20   # stands for a device buffer: no kernel runs

def scene(n=20_000, degree=0, fmt=S.FP32):
    nbytes = S.words_for_degree(degree) * n * (4 if fmt == S.FP32 else 2)
    return G.gs_load_scene(np.zeros(nbytes, np.uint8), n, degree, fmt)

def cams(*sizes):
    return np.concatenate([S.ring_cameras(1, w, h) for w, h in sizes])

def clean(h=None):
    if h is not None:
        G.gs_free_scene(h)
    assert L.fake_report() == b"", L.fake_report().decode()
"""


def run(fake, body):
    code = PRELUDE.format(lib=fake) + textwrap.dedent(body)
    r = subprocess.run([sys.executable, "-c", code], capture_output=True, text=True, timeout=300,
                       cwd=os.path.dirname(HERE))
    assert r.returncode == 0, r.stdout + r.stderr


@pytest.mark.parametrize("first,second", [((1600, 1040), (2592, 1944)), ((2592, 1944), (1600, 1040)),
                                          ((1920, 1080), (2560, 1440)), ((320, 240), (1600, 1040))])
@pytest.mark.parametrize("tile", [(16, 16), (8, 8)])
def test_full_rerender_over_views_of_different_sizes(fake, first, second, tile):
    """Every view's lists are made in tables that hold them: grids on both sides of the
    counting lists' limit, in both orders, at pair capacities that single upsets and
    thousands of upsets a variant ask for."""
    run(fake, f"""
    h = scene()
    G.gs_set_tile(h, *{tile}, stream=0)
    L.fake_counts(2_000_000, 20, 100)
    G.gs_set_views(h, cams({first}, {second}), stream=0)
    for flips in (1, 1000, 5000):
        G.gs_inject_and_render_full(h, ADDR, 2, flips, -1, 0, ADDR, stream=0)
    clean(h)
    """)


def test_counting_tables_hold_every_grid(fake):
    """Tile grids from one tile to past the counting lists' limit, pair capacities from
    one to two billion; a smaller grid after a larger one in the same scratch."""
    run(fake, """
    from itertools import product
    total = np.zeros(1, np.uint64)
    for (tx, ty), cap in product([(1, 1), (7, 1), (9, 9), (50, 50), (100, 65), (69, 100), (83, 83), (139, 100), (140, 100)],
                                 [1, 1000, 1536, 2049, 300_000, 5_000_000, 40_000_000, 2_000_000_000]):
        L.fake_counts(min(cap, 1000), 0, 100)
        G.gs_bin_tiles(ADDR, ADDR, 1, tx, ty, ADDR, ADDR, cap, stream=0)
    for n in (400_000, 1_200_000):
        h = scene(n=n)
        L.fake_counts(9_000_000, 0, 100)
        for W, H in ((2200, 1600), (640, 480), (16, 16), (1600, 1040), (100, 1600), (2592, 1944), (1900, 1250), (800, 800)):
            G.gs_render(h, cams((W, H)), ADDR, stream=0)
        clean(h)
    """)


def test_scratch_after_a_failed_growth(fake):
    """A slot's scratch fails to grow for a large scene, at any of its allocations; the
    next request, of a small one, is given live arrays, and nothing is freed twice."""
    run(fake, """
    for grid in ((640, 480), (2592, 1944)):
        for extra in [0, 1 << 20] + [m << 21 for m in range(1, 90)]:
            small, big = scene(n=5000), scene(n=600_000)
            srv = G.gs_server_create(1 << 40, 1)
            ids = [G.gs_server_add_scene(srv, h) for h in (small, big)]

            def render(i, size, pairs):
                L.fake_counts(pairs, 0, 100)
                t = G.gs_server_submit(srv, G.make_request(G.GS_REQ_RENDER, ids[i], cams(size)[0], dev_rgb=ADDR))
                G.gs_server_wait(srv, t)

            render(0, (640, 480), 9000)
            L.fake_limit(L.fake_live() + extra)
            try:
                render(1, grid, 3_000_000)
            except G.GsError as e:
                assert e.status == G.GS_ERR_OOM, e
            L.fake_limit((1 << 64) - 1)
            render(0, (640, 480), 9000)
            render(0, (2592, 1944), 20_000)
            G.gs_server_destroy(srv)
            G.gs_free_scene(big)
            clean(small)
            assert L.fake_live() == 0
    """)


def test_boxes_after_a_failed_upload(fake):
    """Per-primitive boxes of which only one half found room are no boxes."""
    run(fake, """
    h = scene()
    box = np.zeros(14 * 20_000, np.uint32)
    G.gs_set_prim_box(h, box, box, 14)
    G.gs_set_views(h, cams((320, 240)), stream=0)
    for extra in (0, box.nbytes // 2, box.nbytes):   # on top of the boxes that are replaced
        L.fake_limit(L.fake_live() - 2 * box.nbytes + extra)
        for call in (lambda: G.gs_set_prim_box(h, box, box, 14),
                     lambda: G.gs_inject_and_render(h, ADDR, 8, 1, G.GS_GUARD_PRIM, 1, ADDR, stream=0),
                     lambda: G.gs_guard(h, G.GS_GUARD_PRIM, 1, stream=0)):
            try:
                call()
                raise SystemExit("accepted")
            except G.GsError as e:
                assert e.status in (G.GS_ERR_OOM, G.GS_ERR_STATE, G.GS_ERR_ARG), e   # as with no boxes
        L.fake_limit((1 << 64) - 1)
        G.gs_set_prim_box(h, box, box, 14)
        G.gs_inject_and_render(h, ADDR, 8, 1, G.GS_GUARD_PRIM, 1, ADDR, stream=0)
    clean(h)
    """)


SMALL = 1 << 20   # counters, cameras and the like, that the account leaves out


@pytest.mark.parametrize("sizes", [((1600, 1040),), ((2592, 1944), (640, 480))])
def test_server_account(fake, sizes):
    """The server's resident bytes are the memory that its scenes hold, campaigns'
    batch buffers included; a tight budget holds, and what a campaign grew by is given
    back to a render that waits."""
    run(fake, f"""
    small = {SMALL}
    L.fake_counts(100_000, 30, 100)   # five tiles a primitive: within what a render is admitted for
    h = scene()
    G.gs_set_views(h, cams(*{sizes}), stream=0)
    scene_live = L.fake_live()

    def check(srv, slack=small):
        s = G.gs_server_stats(srv)
        assert abs(s["resident"] + s["scratch"] - L.fake_live()) < slack, (s, L.fake_live())
        return s

    def ask(srv, **kw):
        G.gs_server_wait(srv, G.gs_server_submit(srv, G.make_request(**kw)))

    campaign = dict(kind=G.GS_REQ_CAMPAIGN, scene=0, dev_flips=ADDR, nflips=20_000, dev_results=ADDR)
    render = dict(kind=G.GS_REQ_RENDER, scene=0, cam=cams((1600, 1040))[0], dev_rgb=ADDR)
    srv = G.gs_server_create(1 << 40, 1)
    G.gs_server_add_scene(srv, h)
    check(srv)
    ask(srv, **campaign)
    big = check(srv)["resident"]
    assert big > scene_live + (100 << 20)
    before = L.fake_live()
    ask(srv, **render)
    s = G.gs_server_stats(srv)
    assert s["scratch"] >= L.fake_live() - before > 0   # reserved by its estimate
    scratch = s["scratch"]
    G.gs_server_destroy(srv)
    G.gs_free_scene(h)
    assert L.fake_live() < small

    h = scene()
    G.gs_set_views(h, cams(*{sizes}), stream=0)
    budget = L.fake_live() + scratch + (40 << 20)
    srv = G.gs_server_create(budget, 1)
    G.gs_server_add_scene(srv, h)
    for _ in range(3):
        ask(srv, **campaign)
        s = check(srv, small + scratch)
        assert s["resident"] + s["scratch"] <= budget and L.fake_live() <= budget + small
        ask(srv, **render)
        s = G.gs_server_stats(srv)
        assert s["resident"] + s["scratch"] <= budget and L.fake_live() <= budget + small
    G.gs_server_destroy(srv)
    clean(h)
    """)


def test_batch_size_settles(fake):
    """Where memory is short for the whole batch, a campaign settles for a smaller one:
    the next calls of its size allocate nothing, and the whole batch is back once there
    is memory."""
    run(fake, """
    L.fake_counts(100_000, 30, 100)
    h = scene()
    G.gs_set_views(h, cams((1600, 1040)), stream=0)
    held = L.fake_live()

    def campaign(B=20_000):
        a = L.fake_allocations()
        G.gs_inject_and_render(h, ADDR, B, 1, -1, 0, ADDR, stream=0)
        return L.fake_allocations() - a

    for room in (40 << 20, 300 << 20, 1 << 30):
        G.gs_set_views(h, cams((1600, 1040)), stream=0)
        L.fake_limit(held + room)
        campaign()
        assert held + room // 4 < L.fake_live() <= held + room   # about as much as there is room for
        assert campaign() == 0 and campaign() == 0
        L.fake_limit((1 << 64) - 1)
        assert campaign() > 0 and L.fake_live() > held + (2 << 30)
        assert campaign() == 0
        G.gs_free_scene(h)
        h = scene()
    clean(h)
    """)


@pytest.mark.parametrize("room", [60, 100, 105, 150, 400])
def test_lists_leave_room(fake, room):
    """Blend lists take a view's share of what is free: several views of long lists are
    set where memory holds a part of them only (room: percent of one view's lists)."""
    run(fake, f"""
    n_lists = 200
    L.fake_counts(100_000, n_lists, 1000)
    npix = 1600 * 1040
    h = scene()
    L.fake_limit(L.fake_live() + (400 << 20) + npix * 24 * n_lists * {room} // 100)
    G.gs_set_views(h, cams(*[(1600, 1040)] * 3), stream=0)
    G.gs_inject_and_render(h, ADDR, 20_000, 1, -1, 0, ADDR, stream=0)
    G.gs_render(h, cams((1600, 1040)), ADDR, stream=0)
    clean(h)
    """)


PAIR_STREAM = """
#include <cstdio>
#include "gs_internal.h"
int main() {
    const uint32_t totals[] = {0u, 1u, 63u, 12250000u, 4294000000u, 4294967200u, 4294967231u, 4294967294u};
    for (uint32_t total : totals)
        for (uint32_t runs : {1u, 7u, 1824u, 2432u, 572664u}) {
            uint32_t at = 0;
            for (uint32_t w = 0; w < runs; w++) {   // the runs follow one another and end at the total
                uint32_t p0, p1;
                gs::pair_run(total, runs, w, p0, p1);
                if (p0 != at || p1 < p0) return printf("run %u of %u over %u: %u %u\\n", w, runs, total, p0, p1), 1;
                at = p1;
            }
            if (at != total) return printf("%u of %u pairs in %u runs\\n", at, total, runs), 1;
        }
    for (uint32_t end : {1u, 64u, 65u, 1000u, 4294967231u, 4294967232u, 4294967233u, 4294967294u})
        for (uint32_t first = end > 200u ? end - 200u : 0u; first < end; first++) {
            uint32_t b = first, n = 1;
            while (gs::pair_next(b, end) && n < 10u) n++;
            if (n != (end - first + 63u) / 64u || end - b > 64u) return printf("%u ... %u: %u steps\\n", first, end, n), 1;
        }
    return 0;
}
"""


def test_pair_stream_up_to_32_bits(tmp_path):
    src, exe = tmp_path / "pairs.cu", tmp_path / "pairs"
    src.write_text(PAIR_STREAM)
    cmd = [buildlib.nvcc(), *buildlib.ARCH, "-std=c++17", "-I", buildlib.CSRC, str(src), "-o", str(exe)]
    r = subprocess.run(cmd, capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0, r.stdout

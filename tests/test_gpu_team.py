"""Small images are updated by teams of 16, 8 or 4 warps per 32 pixels
(amh_team.cuh), larger ones and every batch by one thread per pixel: the two
must give the same bits, at the edges of the team's tiles, for the fewest and
the most sources, before and from t = 3 on (one and six refinement
candidates), and for every image form."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

KEYS = ("plane", "cost", "sel", "vbest", "wmask", "choice")


@pytest.fixture(scope="module")
def amh():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1805_07920_gb300 import amh as m
    m.lib()
    return m


def _compare(amh, cams, images, refs, srcs, iters, seed=11, flags=0, **kw):
    P = lambda s: amh.default_params(depth_min=2.0, depth_max=8.0, seed=s, flags=flags, **kw)
    b = amh.Batch(cams, images, refs, srcs, P(seed))
    b.init_random()
    b.iterate(iters)
    for i, (r, src) in enumerate(zip(refs, srcs)):
        g = amh.Context(cams, images, r, src, P(seed + i))
        g.init_random()
        g.iterate(iters)
        g.synchronize()
        one, bat = g.get_state(), b.get_state(i)
        for k in KEYS:
            np.testing.assert_array_equal(one[k], bat[k], err_msg=f"{one['cost'].shape} sources {len(src)} {k}")


# (width, height): one lane, a row, a column, one tile short and past, and the
# sizes that take 16, 8 and 4 warps (96 x 72, 200 x 150, 320 x 200: 108, 494 and
# 1000 tiles of 16 x 4)
@pytest.mark.parametrize("form", ["uint8", "f16", "filter"])
def test_team_sizes(amh, synth_mod, form):
    sizes = [(1, 1), (15, 3), (16, 4), (17, 5), (3, 40), (96, 72), (200, 150), (320, 200)]
    ring = synth_mod.scene_ring20(seed=5, n=8, n_src=3, sizes=sizes)
    images = [im.astype(np.float16) for im in ring.images] if form == "f16" else ring.images
    flags = amh.AMH_FLAG_TEXTURE_BILINEAR if form == "filter" else 0
    _compare(amh, ring.cams, images, list(range(8)), [synth_mod.ring_sources(r, 8, 3) for r in range(8)], 4, flags=flags)


@pytest.mark.parametrize("n_src,k", [(1, 4), (2, 1), (31, 4), (32, 32)])
def test_team_sources(amh, synth_mod, n_src, k):
    sc = synth_mod.scene_many(seed=7)
    _compare(amh, sc.cams, sc.images, [sc.ref], [sc.src[:n_src]], 4, k=k)


def test_team_launches_in_a_graph(amh, synth_mod):
    """The overlapped launches of small images under stream capture: replays of
    the captured initialisation and iterations equal direct calls."""
    import ctypes
    import torch
    sc = synth_mod.make_scene("tiny")
    g = amh.Context.from_scene(sc, seed=21)
    g.init_random()
    g.iterate(4)
    want = g.get_state()
    s = torch.cuda.Stream()
    g.set_stream(ctypes.c_void_p(s.cuda_stream))
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=s):
        g.init_random()
        g.iterate(4)
    for _ in range(2):
        graph.replay()
        torch.cuda.synchronize()
        got = g.get_state()
        for k in KEYS:
            np.testing.assert_array_equal(got[k], want[k], err_msg=k)

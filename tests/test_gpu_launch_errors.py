"""A launch that the CUDA runtime refuses is reported by the call that made it.
The refusal is a host-side one: the stream's capture has been invalidated (by a
synchronisation, which capture forbids), and every launch into it fails until
the capture ends."""
import ctypes

import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("size", [(64, 48), (800, 600)])      # a team of warps and one thread per pixel
def test_refused_launch_is_reported(synth_mod, size):
    import torch
    from paper_1805_07920_gb300 import amh
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    cu = ctypes.CDLL("libcuda.so.1")
    sc = synth_mod.scene_ring20(seed=5, n=3, n_src=2, sizes=[size] * 3)
    s = torch.cuda.Stream()
    h = ctypes.c_void_p(s.cuda_stream)
    g = amh.Context(sc.cams, sc.images, 0, [1, 2], amh.default_params(depth_min=2.0, depth_max=8.0), stream=h)
    g.init_random()
    g.iterate(1)
    want = g.get_state()
    torch.cuda.synchronize()
    assert cu.cuStreamBeginCapture_v2(h, 1) == 0               # thread-local mode
    try:
        assert cu.cuStreamSynchronize(h) != 0                  # not allowed: invalidates the capture
        for call in (g.init_random, lambda: g.step_phase(0)):
            with pytest.raises(amh.AmhError):
                call()
    finally:
        graph = ctypes.c_void_p()
        assert cu.cuStreamEndCapture(h, ctypes.byref(graph)) != 0
    g.init_random()                                            # and the context goes on
    g.iterate(1)
    assert (g.get_state()["plane"] == want["plane"]).all()

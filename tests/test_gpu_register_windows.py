"""The filter form with the window weights in registers (images whose blocks fit
in one or two rounds at three per SM) against the batch, which keeps them in
shared memory: the same bits, up to t = 3, at ragged sizes."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("size,n_src", [((337, 253), 1), ((337, 253), 3), ((521, 391), 6), ((533, 377), 32)])
def test_register_windows(synth_mod, size, n_src):
    import torch
    from paper_1805_07920_gb300 import amh
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    ring = synth_mod.scene_ring20(seed=4, n=n_src + 1, n_src=n_src, sizes=[size] * (n_src + 1))
    src = list(range(1, n_src + 1))
    P = lambda: amh.default_params(depth_min=2.0, depth_max=8.0, seed=5, flags=amh.AMH_FLAG_TEXTURE_BILINEAR)
    b, g = amh.Batch(ring.cams, ring.images, [0], [src], P()), amh.Context(ring.cams, ring.images, 0, src, P())
    for x in (b, g):
        x.init_random()
        x.iterate(5)
        x.synchronize()
    one, bat = g.get_state(), b.get_state(0)
    for k in ("plane", "cost", "sel", "vbest", "wmask", "choice"):
        np.testing.assert_array_equal(one[k], bat[k], err_msg=k)

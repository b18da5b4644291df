"""Every width of the update's teams (amh_update_warps: 16, 8, 4 warps per 32
pixels) and one thread per pixel against the batch, which always takes one
thread per pixel: the same bits for every image form, with few and many sources,
up to t = 3 (one and six refinement candidates), at the largest ragged image
that the device gives each width and the smallest that it gives one thread."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

KEYS = ("plane", "cost", "sel", "vbest", "wmask", "choice")


def _size(amh, n_src, n_sm, warps):
    sizes = [(w, int(w * 0.73) | 1) for w in range(19, 700, 6)]
    fit = [s for s in sizes if amh.update_warps(*s, n_src, n_sm)[1] == warps]
    return (fit[0] if warps == 1 else fit[-1]) if fit else None


@pytest.mark.parametrize("n_src", [1, 3, 5, 32])
@pytest.mark.parametrize("warps", [16, 8, 4, 1])
def test_widths_agree(synth_mod, warps, n_src):
    import torch
    from paper_1805_07920_gb300 import amh
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    n_sm = torch.cuda.get_device_properties(0).multi_processor_count
    size = _size(amh, n_src, n_sm, warps)
    assert size and amh.update_warps(*size, n_src, n_sm)[1] == warps
    ring = synth_mod.scene_ring20(seed=9, n=n_src + 1, n_src=n_src, sizes=[size] * (n_src + 1))
    src = list(range(1, n_src + 1))
    for form in ("uint8", "f16", "filter"):
        images = [im.astype(np.float16) for im in ring.images] if form == "f16" else ring.images
        P = lambda: amh.default_params(depth_min=2.0, depth_max=8.0, seed=3,
                                       flags=amh.AMH_FLAG_TEXTURE_BILINEAR if form == "filter" else 0)
        b = amh.Batch(ring.cams, images, [0], [src], P())
        g = amh.Context(ring.cams, images, 0, src, P())
        for x in (b, g):
            x.init_random()
            x.iterate(4)
            x.synchronize()
        one, bat = g.get_state(), b.get_state(0)
        for k in KEYS:
            np.testing.assert_array_equal(one[k], bat[k], err_msg=f"{size} {form} {k}")

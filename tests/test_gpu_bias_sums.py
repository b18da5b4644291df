"""Rounding of the bias gradients: each is the sum of an FP32 gradient tensor
over the pixels, and the tensor itself can be read, so the sum's own error is
seen.  Targets far below the output give every pixel the same loss gradient, so
each layer sums long runs of equal values, which round the same way everywhere.
A balanced tree of some 16 levels leaves 0.3 * sqrt(16) = 1.2 units of 2^-24 of
the summed magnitudes if each level's additions all round alike (rms over the
channels); 2 is allowed.  A running sum over all of a block's tiles leaves ten
and more."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("w2,h2", [(64, 40), (800, 528), (1600, 1056)])
def test_bias_gradients_round_like_a_tree(w2, h2):
    import torch
    from paper_1805_07920_gb300 import amh
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    layers = [name for name, _, _ in amh.NET_LAYERS if name != "out"]     # summed in the data gradients' epilogues
    rms = {name: [] for name in layers}
    for seed in range(3):
        r = np.random.default_rng(seed)
        net = amh.Net(w2, h2)
        net.set_params({name: (r.normal(0, np.sqrt(2 / (9 * cin)) * (0.1 if name == "out" else 1), (9, cout, cin)).astype(np.float32),
                               r.normal(0, 0.02, cout).astype(np.float32)) for name, cin, cout in amh.NET_LAYERS})
        net.set_example(r.normal(0, 0.4, (h2, w2, 6)).astype(np.float32), np.full((h2, w2, 4), -100, np.float32),
                        np.ones((h2, w2), np.uint8))
        net.forward()
        net.backward()
        grads = net.get_grads()
        for name in layers:
            dy = net.read("dy:" + name).astype(np.float64)
            size = np.abs(dy).sum((0, 1))
            err = np.abs(grads[name][1] - dy.sum((0, 1)))[size > 0] / size[size > 0] * 2.0 ** 24
            rms[name].append(np.sqrt((err ** 2).mean()))
    rms = {name: float(np.mean(v)) for name, v in rms.items()}
    assert max(rms.values()) < 2.0, rms

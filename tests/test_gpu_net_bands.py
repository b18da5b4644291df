"""The network's output to pinned host memory is computed and copied in bands of
rows (the last two layers), to pageable memory in one piece: the same values, for
sizes of one to four bands and rows that end inside a 128-pixel tile."""
import ctypes

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def amh():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1805_07920_gb300 import amh as m
    m.lib()
    return m


@pytest.mark.parametrize("w2,h2", [(8, 8), (72, 40), (136, 64), (264, 104), (128, 136)])
def test_output_bands(amh, w2, h2):
    import torch
    net = amh.Net(w2, h2, seed=5)
    net.set_input(np.random.default_rng(w2).normal(0, 0.5, (h2, w2, 16)))
    whole = net.forward(want_output=True)
    pinned = torch.full((h2, w2, 16), float("nan"), pin_memory=True)
    for _ in range(2):
        net._check(amh.lib().amh_net_forward(net.ctx, ctypes.c_void_p(pinned.data_ptr())))
        np.testing.assert_array_equal(pinned.numpy(), whole)
    np.testing.assert_array_equal(net.read("out"), whole)
    d1 = net.read("d1")
    net.forward()
    np.testing.assert_array_equal(net.read("d1"), d1)

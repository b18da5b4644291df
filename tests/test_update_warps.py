"""Which images are updated by teams of warps (host arithmetic, no GPU)."""
import pytest

from paper_1805_07920_gb300 import amh


@pytest.fixture(scope="module", autouse=True)
def built():
    import os
    from paper_1805_07920_gb300 import _build
    if not os.path.exists(amh.LIB_PATH) or not hasattr(amh.lib(), "amh_update_warps"):
        _build.build()


@pytest.mark.parametrize("n_src", [1, 2, 3, 4, 6, 8, 32])
@pytest.mark.parametrize("n_sm", [78, 148, 152])
def test_rule(n_src, n_sm):
    warps = 16 * n_sm
    last = (16, 16)
    for w in range(16, 1200, 8):
        h = max(4, w * 3 // 4 // 4 * 4)
        groups = (w + 7) // 8 * ((h + 3) // 4), (w + 15) // 16 * ((h + 3) // 4)
        got = amh.update_warps(w, h, n_src, n_sm)
        for g, t, before in zip(groups, got, last):
            assert t in (16, 8, 4, 1) and t <= before              # larger images never take more
            if t > 4:
                assert g * t <= warps                              # all teams at once
        # teams of four that have to take turns lose with one source (240x180 on 152 SMs: 297 us
        # against 277), and with fewer than four in the initialisation (200x150: 10.3 against 8.2)
        if got[1] == 4 and n_src == 1:
            assert groups[1] * 4 <= warps
        if got[0] == 4 and n_src < 4:
            assert groups[0] * 4 <= warps
        last = got
    assert last == (1, 1)


def test_refused():
    for bad in [(0, 4, 1, 152), (4, 0, 1, 152), (4, 4, 0, 152), (4, 4, 33, 152), (4, 4, 1, 0)]:
        with pytest.raises(amh.AmhError):
            amh.update_warps(*bad)
    assert amh.update_warps(32768, 32768, 1, 152) == (1, 1)

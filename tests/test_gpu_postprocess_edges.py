"""Edges of the post-processing kernels: the 4x4 median at the ends of its
29-column strips and 16-row bands, with infinities and NaN; the fusion on views
of uneven sizes whose rows end inside a warp, with thresholds that accept or
refuse everything."""
import numpy as np
import pytest

from oracle import fusion as F

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def amh():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1805_07920_gb300 import amh as m
    m.lib()
    return m


def _sorted_median(d):
    """The windows sorted by the comparisons of an insertion sort (fmin / fmax:
    a NaN gives way to the other operand)."""
    H, W = d.shape
    ys, xs = np.arange(H), np.arange(W)
    v = [d[np.clip(ys + dy, 0, H - 1)][:, np.clip(xs + dx, 0, W - 1)] for dy in (-2, -1, 0, 1) for dx in (-2, -1, 0, 1)]
    for a in range(1, 16):
        for b in range(a, 0, -1):
            v[b - 1], v[b] = np.fmin(v[b - 1], v[b]), np.fmax(v[b - 1], v[b])
    with np.errstate(invalid="ignore"):
        return np.float32(0.5) * v[7] + np.float32(0.5) * v[8]


@pytest.mark.parametrize("shape", [(1, 1), (2, 28), (16, 29), (17, 30), (15, 58), (33, 59), (48, 116), (70, 33)])
@pytest.mark.parametrize("special", [False, True])
def test_median4_edges(amh, shape, special):
    import torch
    r = np.random.default_rng(shape[0] * 131 + shape[1])
    d = r.uniform(0.5, 9, shape).astype(np.float32)
    d[r.random(shape) < 0.2] = np.float32(2.5)            # repeated values
    if special:
        u = r.random(shape)
        d[u < 0.05] = np.inf
        d[(u > 0.05) & (u < 0.1)] = -np.inf
        d[u > 0.97] = np.nan
    got = amh.median4(torch.from_numpy(d).cuda()).cpu().numpy()
    np.testing.assert_array_equal(got, _sorted_median(d))


@pytest.mark.parametrize("kw", [dict(), dict(f_eps=1e9, f_ang_deg=180.0, f_con=1),
                                dict(f_eps=2.0, f_ang_deg=0.0, f_con=1)])
def test_fusion_uneven_views(amh, synth_mod, kw):
    import torch
    sizes = [(33, 17), (64, 9), (31, 40), (1, 1), (95, 66)]
    cams, D, N = [], [], []
    r = np.random.default_rng(3)
    for i, (w, h) in enumerate(sizes):
        R, t = synth_mod.look_at((0.4 * i - 0.8, 0.1 * i, -4.0), (0.0, 0.0, 0.0))
        cams.append(synth_mod.Camera(synth_mod.intrinsics(w, h, 0.9 * max(w, 8)), R, t, w, h))
        y, x = np.mgrid[0:h, 0:w].astype(np.float64)
        ray = np.stack([x, y, np.ones_like(x)], -1) @ np.linalg.inv(cams[-1].K).T
        n = R @ np.array([0.0, 0.0, -1.0])                # the plane z = 0 of the world, in camera coordinates
        d = (n @ (R @ np.zeros(3) + t)) / (ray @ n)
        d = d * (1 + 0.002 * r.standard_normal(d.shape))
        d[r.random(d.shape) < 0.05] = 0.0
        m = n + 0.05 * r.standard_normal((h, w, 3))
        D.append(d.astype(np.float32))
        N.append((m / np.linalg.norm(m, axis=-1, keepdims=True)).astype(np.float32))
    pts, cnt = amh.fuse(cams, [torch.from_numpy(d).cuda() for d in D], [torch.from_numpy(m).cuda() for m in N], **kw)
    opts, oval, ocnt, amb = F.fuse(cams, D, N, **kw)
    for v in range(len(sizes)):
        clear = ~amb[v]
        np.testing.assert_array_equal(cnt[v].cpu().numpy()[clear], ocnt[v][clear], err_msg=f"view {v}")
        p = pts[v].cpu().numpy()
        both = clear & oval[v]
        assert np.abs(p[both] - opts[v][both]).max(initial=0.0) < 1e-3
        assert not p[clear & ~oval[v]].any()

"""Fusion decisions at their boundaries.  Away from them the kernel decides by
hardware estimates; next to them it repeats the check with correctly rounded
quotients and roots.  Here every product and sum is exact in FP32 (identity
rotations, a focal length of 64, integer translations, depths and normals), so
only the quotients and roots round and NumPy's FP32 gives the one right answer:
images exactly on a half pixel and one unit beside it, disparities at f_eps and
one unit in the last place beside it, angles likewise.  No pixel is left out."""
import math

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

F32 = np.float32
W, H, FOCAL, CX, CY = 128, 48, 64, 64, 24
SHIFT = 384                                   # camera offset: an image moves by 64 x 384 / depth pixels
HALF = 2 * FOCAL * SHIFT                      # the depth at which that is half a pixel
T = [(0, 0, 0), (SHIFT, 0, 0), (-SHIFT, SHIFT, 0)]


def _maps(seed):
    r = np.random.default_rng(seed)
    depths = np.array([HALF, HALF - 1, HALF + 1, HALF - 2, HALF + 2, HALF - 3, HALF // 3, HALF // 3 + 1, 0])
    normals = np.array([(3, 4, 12), (4, 3, 12), (12, 3, 4), (-3, 4, 12), (1, 2, 3), (2, 1, 3), (0, 0, -1)])
    D = [r.choice(depths, (H, W), p=[.2, .15, .15, .12, .12, .1, .07, .04, .05]).astype(F32) for _ in T]
    N = [normals[r.integers(0, len(normals), (H, W))].astype(F32) for _ in T]
    return D, N


def _fuse32(D, N, eps, cos_ang):
    """(points, counts, decisions within the estimates' error of a boundary, of
    the pixel / the disparity / the angle)."""
    y, x = np.mgrid[0:H, 0:W].astype(F32)
    f, eps, cos_ang = F32(FOCAL), F32(eps), F32(cos_ang)
    out, near = [], np.zeros(3, int)
    world = lambda d, px, py, t: [d * ((px - F32(CX)) / f) - F32(t[0]), d * ((py - F32(CY)) / f) - F32(t[1]), d - F32(t[2])]
    for i, ti in enumerate(T):
        z = D[i]
        has = z > 0
        sX, sN, cnt = world(z, x, y, ti), [N[i][..., k].copy() for k in range(3)], np.zeros((H, W), np.uint8)
        X = [a.copy() for a in sX]
        nn = np.sqrt((N[i] * N[i]).sum(-1))
        for j, tj in enumerate(T):
            if j == i:
                continue
            with np.errstate(divide="ignore", invalid="ignore"):
                u = (f * (X[0] + F32(tj[0])) + F32(CX) * z) / z
                v = (f * (X[1] + F32(tj[1])) + F32(CY) * z) / z
            u, v = np.where(has, u, F32(-9)), np.where(has, v, F32(-9))
            uf, vf = np.floor(u + F32(.5)), np.floor(v + F32(.5))
            ins = has & (uf >= 0) & (uf < W) & (vf >= 0) & (vf < H)
            q = np.where(ins, vf, 0).astype(int), np.where(ins, uf, 0).astype(int)
            Dj, Nj = D[j][q], N[j][q]
            ok = ins & (Dj > 0)
            one = np.where(ok, Dj, F32(1)), np.where(has, z, F32(1))
            wb = f * np.sqrt(F32(sum((a - b) ** 2 for a, b in zip(ti, tj))))
            disp = wb * np.abs(F32(1) / one[1] - F32(1) / one[0])
            cosine = (N[i] * Nj).sum(-1) / np.maximum(np.sqrt((Nj * Nj).sum(-1)) * nn, F32(1e-30))
            agree = ok & (disp <= eps) & (cosine >= cos_ang)
            near[0] += (has & (np.maximum(np.abs(u - uf), np.abs(v - vf)) > 0.5 - 2.0 ** -21 * (1 + np.maximum(abs(u), abs(v))))).sum()
            near[1] += (ok & (np.abs(disp - eps) <= 2.0 ** -22 * wb * (1 / one[0] + 1 / one[1]))).sum()
            near[2] += (ok & (disp <= eps) & (np.abs(cosine - cos_ang) <= 4e-6)).sum()
            for k, a in enumerate(world(Dj, uf, vf, tj)):
                sX[k] = np.where(agree, sX[k] + a, sX[k])
                sN[k] = np.where(agree, sN[k] + Nj[..., k], sN[k])
            cnt += agree
        ln = np.maximum(np.sqrt(sN[0] * sN[0] + sN[1] * sN[1] + sN[2] * sN[2]), F32(1e-30))
        p = np.stack([s * (F32(1) / (1 + cnt).astype(F32)) for s in sX] + [s / ln for s in sN], -1)
        out.append((np.where((has & (cnt >= 1))[..., None], p, F32(0)), np.where(has, cnt, 0).astype(np.uint8)))
    return out, near


def _angle(cos_ang):
    """An FP32 angle in degrees whose cosine, as the library computes it, rounds to cos_ang."""
    a = F32(math.degrees(math.acos(min(1.0, float(cos_ang)))))
    for _ in range(1000):
        c = F32(math.cos(float(a) * math.pi / 180.0))
        if c == F32(cos_ang):
            return float(a)
        a = np.nextafter(a, F32(0) if c < F32(cos_ang) else F32(180))
    raise AssertionError("no such angle")


# thresholds: the disparity of depths d and d + 1 of views 0 and 1 at half a pixel,
# the cosine of two normals; each one unit in the last place below, there, above
_EPS = F32(FOCAL * SHIFT) * (F32(1) / F32(HALF) - F32(1) / F32(HALF + 1))
_COS = [F32(168) / F32(169), F32(13) / (np.sqrt(F32(14)) * np.sqrt(F32(14)))]


def _steps(a):
    return [np.nextafter(a, F32(0)), a, np.nextafter(a, F32(2))]


CASES = ([(e, F32(0.5)) for e in _steps(_EPS)] + [(F32(1), c) for k in _COS for c in _steps(k)] +
         [(F32(0), F32(0.5)), (F32(1), F32(1))])


@pytest.mark.parametrize("case", range(len(CASES)))
def test_decisions_at_their_boundaries(synth_mod, case):
    import torch
    from paper_1805_07920_gb300 import amh
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    eps, cos_ang = CASES[case]
    D, N = _maps(case)
    ang = _angle(cos_ang)
    want, near = _fuse32(D, N, eps, F32(math.cos(ang * math.pi / 180.0)))
    assert near[0] > 1000 and near[1 if eps < F32(1) else 2] > 1000, near
    K = np.array([[FOCAL, 0, CX], [0, FOCAL, CY], [0, 0, 1]], float)
    cams = [synth_mod.Camera(K, np.eye(3), np.array(t, float), W, H) for t in T]
    pts, cnt = amh.fuse(cams, [torch.from_numpy(d).cuda() for d in D], [torch.from_numpy(n).cuda() for n in N],
                        f_eps=float(eps), f_ang_deg=ang, f_con=1)
    for v, (p, c) in enumerate(want):
        np.testing.assert_array_equal(cnt[v].cpu().numpy(), c, err_msg=f"view {v}")
        np.testing.assert_array_equal(pts[v].cpu().numpy(), p, err_msg=f"view {v}")

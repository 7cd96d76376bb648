"""The bound map is finite where its construction says so and not loose: every texel against a float64
walk of its centre ray through the grid maximised over one layer more than the map's own
neighbourhoods (a ray along a face may take the cells of either side)."""
import numpy as np
import pytest

from paper_2406_15632_gb300 import scenes as S

pytestmark = pytest.mark.gpu

LO, HI = np.array([-1.2, -0.9, -1.0]), np.array([1.0, 1.1, 0.8])


def _directions(m):
    """Unit centre directions [6][m][m][3] and the cosines to the farthest corner."""
    c = (np.arange(m) + 0.5) * (2.0 / m) - 1.0
    v, u = np.meshgrid(c, c, indexing="ij")
    out, cosine = np.empty((6, m, m, 3)), np.ones((6, m, m))
    for f in range(6):
        a = f // 2
        b, k = [q for q in range(3) if q != a]

        def face(uu, vv):
            d = np.empty((m, m, 3))
            d[..., a], d[..., b], d[..., k] = (-1.0 if f % 2 else 1.0), uu, vv
            return d / np.linalg.norm(d, axis=-1, keepdims=True)

        out[f] = face(u, v)
        for su in (-1, 1):
            for sv in (-1, 1):
                cosine[f] = np.minimum(cosine[f], (out[f] * face(u + su / m, v + sv / m)).sum(-1))
    return out, cosine


def _walk(K, lo, h, dirs):
    """Integrals of the cells K (lower corner lo, edges h) along rays from the origin."""
    n = np.array(K.shape[::-1])
    flat = dirs.reshape(-1, 3)
    out = np.empty(len(flat))
    for s in range(0, len(flat), 4096):
        d = flat[s:s + 4096]
        with np.errstate(divide="ignore", invalid="ignore"):
            t = np.concatenate([(lo[a] + h[a] * np.arange(n[a] + 1))[None, :] / d[:, a:a + 1] for a in range(3)], axis=1)
        t = np.sort(np.where(np.isfinite(t) & (t > 0), t, 0.0), axis=1)
        t = np.concatenate([np.zeros((len(d), 1)), t], axis=1)
        mid = 0.5 * (t[:, 1:] + t[:, :-1])
        c = np.floor((mid[..., None] * d[:, None, :] - lo) / h).astype(int)
        ok = ((c >= 0) & (c < n)).all(-1)
        c = np.clip(c, 0, n - 1)
        out[s:s + 4096] = (np.where(ok, K[c[..., 2], c[..., 1], c[..., 0]], 0.0) * np.diff(t, axis=1)).sum(1)
    return out.reshape(dirs.shape[:-1])


@pytest.mark.parametrize("shape,m,star_r", [((4, 4, 4), 9, 0.0), ((3, 5, 7), 31, 0.0), ((33, 17, 30), 64, 0.0),
                                            ((33, 17, 30), 128, 0.0), ((12, 16, 20), 64, 0.1), ((12, 16, 20), 40, 0.3)])
def test_finite_and_tight(shape, m, star_r):
    import torch
    from scipy.ndimage import maximum_filter

    from paper_2406_15632_gb300 import build as B
    from paper_2406_15632_gb300 import qmcrt as Q

    B.build()
    Q.load()
    g = np.random.default_rng(5).uniform(0.0, 2.0, size=shape).astype(np.float32)
    star = dict(source="sphere", star_r=star_r) if star_r else {}
    sky = Q.Scene(S.Problem(grid=g, lo=tuple(LO), hi=tuple(HI), nx=8, ny=8, **star), sky=m, tail=False).sky
    torch.cuda.synchronize()
    sky = sky.cpu().numpy()
    n = np.array(shape[::-1])
    h = (HI - LO) / n
    dirs, cosine = _directions(m)
    R = star_r * (1.0 + 1e-4)
    D = 1 + int(np.ceil(R / h.min()))
    tmax = np.sqrt(((np.maximum(np.abs(LO), np.abs(HI)) + R) ** 2).sum())
    spare = D * h.min() - R - tmax * np.arccos(np.minimum(cosine, 1.0))
    band = 2e-5 * tmax  # of the float angle, its margins and the map's own room
    assert np.isfinite(sky[spare > band]).all()
    assert np.isinf(sky[spare < 0.0]).all()
    assert (spare > band).any()
    K = np.pad(g.astype(np.float64), D + 1)
    K = maximum_filter(K, size=2 * (D + 1) + 1, mode="constant")
    ref = _walk(K, LO - (D + 1) * h, h, dirs)
    fin = np.isfinite(sky)
    assert (sky[fin] <= ref[fin] * 1.001).all()

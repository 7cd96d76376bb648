"""The padded grid, the bound map and the tail map at the sizes where their kernels change form:
rows of whole vectors or not, one to many blocks a thread, slabs too large for shared memory,
boxes one cell thin, offset pointers.  Against plain numpy of the same definitions."""
import math

import numpy as np
import pytest

from paper_2406_15632_gb300 import scenes as S

pytestmark = pytest.mark.gpu

SHAPES = [(4, 4, 4), (1, 1, 1), (3, 5, 7), (8, 9, 33), (17, 16, 30), (31, 29, 64), (1, 2, 61), (64, 12, 4), (40, 40, 40)]


@pytest.fixture(scope="module")
def Q():
    from paper_2406_15632_gb300 import build as B
    from paper_2406_15632_gb300 import qmcrt

    B.build()
    qmcrt.load()
    return qmcrt


def _grid(shape, seed=0):
    rng = np.random.default_rng(seed)
    g = rng.uniform(0.0, 2.0, size=shape).astype(np.float32)
    g[rng.uniform(size=shape) < 0.3] = 0.0
    return g


@pytest.mark.parametrize("pad", [8, 9])
@pytest.mark.parametrize("shape", SHAPES)
def test_padded_copy(Q, shape, pad):
    import torch

    g = _grid(shape)
    g.flat[0] = -3.0
    g.flat[-1] = np.nan
    ref = np.full([n + 2 * pad for n in shape], -0.0, dtype=np.float32)
    ref[pad:-pad, pad:-pad, pad:-pad] = np.where(g > 0, g, 0.0)
    for shift in (0, 1):  # a grid and a copy that do not start on 16 bytes
        src = torch.zeros(g.size + 4, device="cuda")
        src[shift:shift + g.size] = torch.from_numpy(g.ravel()).cuda()
        dst = torch.full((ref.size + 8,), 5.0, device="cuda")
        nz, ny, nx = shape
        Q.qmcrt_pad_grid(src.data_ptr() + 4 * shift, nx, ny, nz, pad, dst.data_ptr() + 4 * shift)
        torch.cuda.synchronize()
        out = dst.cpu().numpy()
        got = out[shift:shift + ref.size]
        assert np.array_equal(got.view(np.uint32), ref.ravel().view(np.uint32))
        assert (out[:shift] == 5.0).all() and (out[shift + ref.size:] == 5.0).all()


def _tail_model(g, lo, hi, k):
    """The slab recurrence of the tail map in float64 (block bounds, no upward rounding)."""
    nz, ny, nx = g.shape
    n = [nx, ny, nz]
    nb = [-(-v // 4) for v in n]
    Kb = np.zeros(nb[::-1])
    for z in range(nb[2]):
        for y in range(nb[1]):
            for x in range(nb[0]):
                Kb[z, y, x] = max(0.0, g[4 * z:4 * z + 4, 4 * y:4 * y + 4, 4 * x:4 * x + 4].max())
    Kb = Kb.transpose(2, 1, 0)  # [x][y][z]
    h = [(hi[q] - lo[q]) / n[q] for q in range(3)]
    speed = [abs(k[q]) / h[q] for q in range(3)]
    a = max(range(3), key=lambda q: (speed[q], -q))
    lat = []
    for q in range(3):
        r = speed[q] / speed[a] * (1 + 1e-9)
        lat.append(1 if q == a or k[q] == 0 else 1 + (3 + math.floor(4 * r) + 2) // 4)
    sgn = [int(np.sign(v)) for v in k]

    def spread(A):  # maximum over the lateral blocks
        out = A.copy()
        for q in range(3):
            src = out.copy()
            for o in range(1, lat[q]):
                sl_to, sl_from = [slice(None)] * 3, [slice(None)] * 3
                sl_to[q] = slice(0, -o) if sgn[q] > 0 else slice(o, None)
                sl_from[q] = slice(o, None) if sgn[q] > 0 else slice(0, -o)
                if src.shape[q] > o:
                    out[tuple(sl_to)] = np.maximum(out[tuple(sl_to)], src[tuple(sl_from)])
        return out

    path = 4 * h[a] / abs(k[a])
    Kl, B = spread(Kb), np.zeros_like(Kb)
    prev = None
    for j in (range(nb[a] - 1, -1, -1) if sgn[a] > 0 else range(nb[a])):
        ix = [slice(None)] * 3
        ix[a] = slice(j, j + 1)
        cur = Kl[tuple(ix)] * path + (0.0 if prev is None else spread(prev))
        B[tuple(ix)] = cur
        prev = cur
    return np.repeat(np.repeat(np.repeat(B, 4, 0), 4, 1), 4, 2)[:nx, :ny, :nz].transpose(2, 1, 0)


@pytest.mark.parametrize("theta,phi", [(0.7, 0.3), (2.2, 4.0), (math.pi / 2, 0.0), (0.0, 0.0), (1.5, -1.2)])
@pytest.mark.parametrize("shape", SHAPES + [(140, 132, 5), (4, 520, 132), (3, 530, 516)])
def test_tail_map_follows_the_slab_recurrence(Q, shape, theta, phi):
    """Codes equal the exponent of the recurrence's bound; upward rounding of float sums and of
    the path (1 + 1e-6 a slab at most) may raise a bound across a power of two."""
    import torch

    g = _grid(shape, 3)
    prob = S.Problem(grid=g, lo=(-1.2, -0.9, -1.0), hi=(1.0, 1.1, 0.8), theta_obs=theta, phi_obs=phi, nx=8, ny=8)
    for pad in (8, 9):
        sc = Q.Scene(prob, pad=pad, tail=True, sky=0)
        torch.cuda.synchronize()
        nz, ny, nx = shape
        m = sc.tail.cpu().numpy().reshape(nz + 2 * pad, ny + 2 * pad, nx + 2 * pad)
        codes = m[pad:-pad, pad:-pad, pad:-pad].astype(int)
        assert m.astype(int).sum() == codes.sum()  # nothing in the padding
        st, ct = math.sin(theta), math.cos(theta)
        B = _tail_model(g, prob.lo, prob.hi, [st * math.cos(phi), st * math.sin(phi), ct])
        want = lambda b: np.where(b > 0, np.frexp(np.maximum(b, 1e-300))[1] - 1 + 127 + 24, 0)
        assert (codes >= want(B)).all()
        assert (codes <= want(B * (1 + 2e-6 * (1 + max(shape) / 4)))).all()


@pytest.mark.parametrize("m", [1, 3, 8, 9, 31, 64])
@pytest.mark.parametrize("shape", [(4, 4, 4), (3, 5, 7), (1, 2, 40), (33, 17, 30)])
def test_bound_map_holds_along_random_rays(Q, shape, m):
    """Every finite texel bounds the optical depth (float64 sums of exact segments) of rays in it."""
    import torch

    g = _grid(shape, 5)
    prob = S.Problem(grid=g, lo=(-1.2, -0.9, -1.0), hi=(1.0, 1.1, 0.8), nx=8, ny=8)
    sc = Q.Scene(prob, sky=m, tail=False)
    torch.cuda.synchronize()
    sky = sc.sky.cpu().numpy()
    assert not np.isnan(sky).any()
    n = np.array(shape[::-1])
    lo, hi = np.array(prob.lo), np.array(prob.hi)
    h = (hi - lo) / n
    rng = np.random.default_rng(m)
    for d in rng.normal(size=(200, 3)):
        d /= np.linalg.norm(d)
        ts = [0.0]
        for a in range(3):
            t = (lo[a] + h[a] * np.arange(n[a] + 1)) / d[a]
            ts += t[t > 0].tolist()
        ts = np.unique(ts)
        mid = 0.5 * (ts[1:] + ts[:-1])[:, None] * d
        c = np.floor((mid - lo) / h).astype(int)
        ok = ((c >= 0) & (c < n)).all(1)
        tau = float(np.sum(g[c[ok, 2], c[ok, 1], c[ok, 0]] * (ts[1:] - ts[:-1])[ok]))
        a = int(np.argmax(np.abs(d)))
        u, v = (d[q] / abs(d[a]) for q in range(3) if q != a)
        iu, iv = (min(m - 1, max(0, int((w + 1) / 2 * m))) for w in (u, v))
        assert tau <= sky[2 * a + (d[a] < 0), iv, iu] * (1 + 1e-12)

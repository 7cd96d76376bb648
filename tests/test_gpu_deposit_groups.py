"""Deposits of warps that hit from one to more pixels than are summed before the atomics: fixed-point
images from few pixels to many, against the sum over the packet log (nearest) and against the FP64
accumulator (both splats)."""
import numpy as np
import pytest

from paper_2406_15632_gb300 import scenes as S

pytestmark = pytest.mark.gpu

FB = 40


@pytest.fixture(scope="module")
def Q():
    from paper_2406_15632_gb300 import build as B
    from paper_2406_15632_gb300 import qmcrt

    B.build()
    qmcrt.load()
    return qmcrt


@pytest.mark.parametrize("source", ["point", "sphere"])
@pytest.mark.parametrize("n", [1, 31, 1000, 40_000])
@pytest.mark.parametrize("nx,ny", [(1, 1), (2, 1), (3, 2), (4, 4), (16, 9), (200, 180)])
def test_images_of_few_and_many_pixels(Q, nx, ny, n, source):
    import torch

    star = dict(source="sphere", star_r=0.2) if source == "sphere" else {}
    p = S.Problem(grid=S.random_grid(8, 1), albedo=0.9, g=0.3, p_l=0.5, theta_obs=1.0, half_width=1.1, nx=nx, ny=ny,
                  **star)
    img, log = Q.render(p, n, first=5, precision="f64", accum="i64", frac_bits=FB, log=True, scale=2.0 ** FB)
    r = log.cpu().numpy()
    r = r[r[:, 8] == 0]
    fx, fy = (np.floor((r[:, 6] + 1.1) * (nx / 2.2)), np.floor((r[:, 7] + 1.1) * (ny / 2.2)))
    ok = (fx >= 0) & (fx < nx) & (fy >= 0) & (fy < ny)
    want = np.zeros((3, ny, nx), np.int64)
    for k in range(3):
        np.add.at(want[k], (fy[ok].astype(int), fx[ok].astype(int)), np.rint(r[ok, 3 + k] * 2.0 ** FB).astype(np.int64))
    assert np.abs(want).max() < 2 ** 53  # the reduced image holds them exactly
    assert np.array_equal(img[0].cpu().numpy(), want.astype(np.float64))
    for splat in ("nearest", "bilinear"):
        q = p.replace(splat=splat)
        a = Q.render(q, n, first=5, precision="f64", accum="i64", frac_bits=FB, scale=1.0)
        b = Q.render(q, n, first=5, precision="f64", accum="f64", scale=1.0)
        # half a unit a deposit, and the FP64 sums' rounding
        assert bool(((a - b).abs() <= 4 * n * (2.0 ** -(FB + 1) + 2.0 ** -52)).all())
    assert n < 1000 or bool((img != 0).any())

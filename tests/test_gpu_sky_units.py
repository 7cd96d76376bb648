"""The bound map does not depend on the unit of length: in a box scaled by a power of two, with
densities scaled back, every texel is the same bit for bit, infinite ones among them."""
import numpy as np
import pytest

from paper_2406_15632_gb300 import scenes as S

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("star_r", [0.0, 0.05])
@pytest.mark.parametrize("n,m", [(64, 80), (64, 120), (250, 320)])
def test_map_of_a_scaled_box(n, m, star_r):
    import torch

    from paper_2406_15632_gb300 import build as B
    from paper_2406_15632_gb300 import qmcrt as Q

    B.build()
    Q.load()
    g = np.random.default_rng(n).uniform(0.1, 2.0, size=(n, n, n)).astype(np.float32)

    def sky(e):
        u = 2.0 ** e
        star = dict(source="sphere", star_r=star_r * u) if star_r else {}
        p = S.Problem(grid=g / np.float32(u), lo=(-1.25 * u, -u, -u), hi=(u, 1.5 * u, u), half_width=u, nx=8, ny=8, **star)
        return Q.Scene(p, sky=m, tail=False).sky

    ref = sky(0)
    assert bool(torch.isfinite(ref).any())
    for e in (-60, -20, -7, 5, 60):
        assert torch.equal(sky(e), ref)

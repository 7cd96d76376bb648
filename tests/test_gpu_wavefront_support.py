"""The wavefront ends walks where they leave the medium's support (a ball and a cylinder around
its nonzero cells); the one-kernel tracer walks to the box's edge.  Images are equal bit for
bit on media whose support is small, off centre, thin along one axis, a single cell, absent or
the whole box, in boxes of unequal edges."""
import numpy as np
import pytest

from paper_2406_15632_gb300 import scenes as S

pytestmark = pytest.mark.gpu


def _medium(name):
    rng = np.random.default_rng(4)
    nz, ny, nx = 22, 19, 25
    z, y, x = np.meshgrid(*(2 * (np.arange(n) + 0.5) / n - 1 for n in (nz, ny, nx)), indexing="ij")
    full = rng.uniform(0.5, 6.0, size=(nz, ny, nx)).astype(np.float32)
    keep = {"ball": x * x + y * y + z * z < 0.3, "column": x * x + y * y < 0.2, "plate": np.abs(z) < 0.15,
            "corner": (x > 0.5) & (y > 0.5) & (z > 0.5), "rod": (np.abs(x) < 0.2) & (np.abs(z) < 0.2),
            "full": np.ones_like(full, bool), "empty": np.zeros_like(full, bool)}
    if name == "cell":
        g = np.zeros_like(full)
        g[14, 6, 20] = 50.0
        return g
    return np.where(keep[name], full, 0).astype(np.float32)


@pytest.fixture(scope="module")
def Q():
    from paper_2406_15632_gb300 import build as B
    from paper_2406_15632_gb300 import qmcrt

    B.build()
    qmcrt.load()
    return qmcrt


@pytest.mark.parametrize("precision", ["f32", "f64"])
@pytest.mark.parametrize("name", ["ball", "column", "plate", "corner", "rod", "full", "empty", "cell"])
def test_walks_ended_at_the_support_change_no_image(Q, name, precision):
    import torch

    prob = S.Problem(grid=_medium(name), lo=(-1.2, -0.9, -2.0), hi=(1.0, 1.1, 1.6), albedo=0.9, g=0.3, p_l=0.4,
                     theta_obs=1.1, phi_obs=0.4, half_width=2.0, nx=30, ny=30, max_orders=6, per_order=True,
                     tau_min=0.0 if name == "rod" else 1e-12)
    sc = Q.Scene(prob)
    a, b = sc.accum_buffer("i64"), sc.accum_buffer("i64")
    n = 20_000
    sc.trace(1, n, a, frac_bits=36, precision=precision)
    sc.trace_wavefront(1, n, b, sc.wavefront_workspace(n, precision), frac_bits=36, precision=precision)
    torch.cuda.synchronize()
    assert torch.equal(a, b)
    assert bool((a != 0).any()) == (name != "empty")

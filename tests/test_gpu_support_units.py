"""Walks that end at the medium's support end at the same cell whatever the unit of length: boxes
of 1e-20 to 1e22 units and edges far apart, and a box that does not hold the origin.  A wavefront's image equals
the one-kernel tracer's bit for bit, a batch's the lone traces'."""
import numpy as np
import pytest

from paper_2406_15632_gb300 import scenes as S

pytestmark = pytest.mark.gpu

N = 24
c = 2 * (np.arange(N) + 0.5) / N - 1
Z, Y, X = np.meshgrid(c, c, c, indexing="ij")
BALL = (X * X + Y * Y + Z * Z < 0.8) * np.random.default_rng(2).uniform(0.5, 4.0, size=(N, N, N))
BOXES = {"1e22": ((-1e22,) * 3, (1e22,) * 3), "3e22": ((-3e22,) * 3, (3e22,) * 3), "1e-20": ((-1e-20,) * 3, (1e-20,) * 3),
         "flat": ((-1.0, -1e3, -1e-2), (1.0, 1e3, 1e-2)),
         "flat 1e18": ((-1e18, -1e21, -1e16), (1e18, 1e21, 1e16)), "needle": ((-1.0, -1.0, -1e8), (1.0, 1.0, 1e8)),
         "slab 3e20": ((-1e20, -3e20, -1e18), (1e20, 3e20, 1e18)), "corner": ((-0.01,) * 3, (1.99,) * 3), "unit": ((-1.0,) * 3, (1.0,) * 3)}


@pytest.fixture(scope="module")
def Q():
    from paper_2406_15632_gb300 import build as B
    from paper_2406_15632_gb300 import qmcrt

    B.build()
    qmcrt.load()
    return qmcrt


def _problem(box, **kw):
    lo, hi = BOXES[box]
    unit = max(hi)
    return S.Problem(grid=(BALL / min(hi)).astype(np.float32), lo=lo, hi=hi, albedo=0.9, g=0.3, p_l=0.4, theta_obs=1.1,
                     phi_obs=0.4, half_width=unit, nx=30, ny=30, **kw)


@pytest.mark.parametrize("box", list(BOXES))
def test_wavefront(Q, box):
    import torch

    sc = Q.Scene(_problem(box, max_orders=5, per_order=True), sky=0)
    a, b = sc.accum_buffer("i64"), sc.accum_buffer("i64")
    n = 20_000
    sc.trace(1, n, a, frac_bits=36, precision="f64")
    sc.trace_wavefront(1, n, b, sc.wavefront_workspace(n, "f64"), frac_bits=36, precision="f64")
    torch.cuda.synchronize()
    assert torch.equal(a, b)
    assert bool((a[:, 1:] != 0).any())


@pytest.mark.parametrize("box", list(BOXES))
def test_batch(Q, box):
    import torch

    p = _problem(box, source="sphere", star_r=0.1 * min(BOXES[box][1]))
    inst = [S.Instance(theta_obs=0.3 * k, albedo=0.7, g=0.4, kscale=0.5 + k, n_packets=4096, first_index=4096)
            for k in range(3)]
    b = Q.Batch(p, inst, precision="f64", frac_bits=36, tails=False)
    b.run()
    got = b.accum.clone()
    b.run_each()
    torch.cuda.synchronize()
    assert torch.equal(got, b.accum)
    assert bool((got != 0).any())


@pytest.mark.parametrize("precision", ["f32", "f64"])
def test_box_beside_the_star(Q, precision):
    """Packets of a large star enter a box on its surface, far from the origin in its edges."""
    import torch

    g = (BALL * 4).astype(np.float32)
    p = S.Problem(grid=g, lo=(29.0, -1.0, -1.0), hi=(31.0, 1.0, 1.0), albedo=0.9, g=0.3, source="sphere", star_r=30.0,
                  theta_obs=1.1, phi_obs=0.4, half_width=40.0, nx=64, ny=64, max_orders=4, per_order=True)
    sc = Q.Scene(p, sky=0)
    a, b = sc.accum_buffer("i64"), sc.accum_buffer("i64")
    n = 1 << 18
    sc.trace(1, n, a, frac_bits=36, precision=precision)
    sc.trace_wavefront(1, n, b, sc.wavefront_workspace(n, precision), frac_bits=36, precision=precision)
    torch.cuda.synchronize()
    assert torch.equal(a, b)
    assert bool((a[:, 1:] != 0).any())


@pytest.mark.parametrize("precision", ["f32", "f64"])
@pytest.mark.parametrize("sizes", [(1,), (5,), (6,), (7,), (2047,), (2048,), (100, 8191), (8192, 0, 5), (0, 0), (700, 700, 700)])
def test_small_batches_with_and_without_the_cut(Q, sizes, precision):
    """Batches on both sides of the size from which the support is looked for, one after another in one
    workspace."""
    import torch

    p = _problem("unit", source="sphere", star_r=0.1)
    sc = Q.Scene(p)
    inst = [S.Instance(theta_obs=0.3 * k, albedo=0.7, g=0.4, kscale=0.5 + k, n_packets=n, first_index=9)
            for k, n in enumerate(sizes)]
    b = Q.Batch(p, inst, frac_bits=36, scene=sc, precision=precision)
    for _ in range(2):
        b.run()
        got = b.accum.clone()
        b.ws.fill_(-1)
    b.run_each()
    torch.cuda.synchronize()
    assert torch.equal(got, b.accum)
    assert bool((got != 0).any()) == (max(sizes) > 0)


@pytest.mark.parametrize("orders,n", [(2, 3), (2, 4), (2, 5), (3, 1), (3, 2), (9, 40)])
def test_short_wavefronts_with_and_without_the_cut(Q, orders, n):
    """Counts on both sides of the one from which a run looks for the support, of a 64^3 grid."""
    import torch

    p = _problem("unit", max_orders=orders, per_order=True)
    p = p.replace(grid=np.repeat(np.repeat(np.repeat(p.grid, 3, 0), 3, 1), 3, 2)[4:68, 4:68, 4:68].copy())
    sc = Q.Scene(p, sky=0)
    a, b = sc.accum_buffer("i64"), sc.accum_buffer("i64")
    sc.trace(7, n, a, frac_bits=36)
    sc.trace_wavefront(7, n, b, sc.wavefront_workspace(n), frac_bits=36)
    torch.cuda.synchronize()
    assert torch.equal(a, b)

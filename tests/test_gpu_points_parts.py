"""Short outputs of many dimensions, whose tiles several blocks share: ranges at the edges of the
parts (32 rows) and around the number of tiles up to which they are shared, bit-exact against the CPU
oracle, with the words around the output untouched."""
import numpy as np
import pytest

from oracle import oracle as O

pytestmark = pytest.mark.gpu

RANGES = [(16, 1, 31), (16, 1, 33), (17, 31, 1), (20, 32, 32), (33, 255, 66), (80, 200, 300), (16, 5, 38 * 256 - 5),
          (16, 5, 38 * 256 - 4), (19, 256, 39 * 256 + 1), (256, 1, 100), (256, 64, 160), (15, 1, 500)]


@pytest.fixture(scope="module")
def Q():
    from paper_2406_15632_gb300 import build as B
    from paper_2406_15632_gb300 import qmcrt

    B.build()
    qmcrt.load()
    return qmcrt


@pytest.mark.parametrize("dims,first,count", RANGES)
@pytest.mark.parametrize("fmt", ["u32", "f32", "f64"])
@pytest.mark.parametrize("kind", ["sobol", "sobol_owen", "niederreiter"])
def test_points_of_shared_tiles(Q, kind, fmt, dims, first, count):
    import torch

    dt = {"u32": torch.int32, "f32": torch.float32, "f64": torch.float64}[fmt]
    for shift in (0, 1):
        buf = torch.full((count * dims + 8,), -7, dtype=dt, device="cuda")
        out = buf[shift:shift + count * dims]
        Q.generate_points(kind, dims, first, count, fmt, seed=77, out=out)
        torch.cuda.synchronize()
        ref = O.generate_points(kind, dims, first, count, fmt, seed=77)
        assert np.array_equal(out.cpu().numpy().reshape(count, dims).view(np.uint8), ref.view(np.uint8))
        assert bool((buf[:shift] == -7).all()) and bool((buf[shift + count * dims:] == -7).all())

"""GPU point sets at the edges of the tiles they are written in (256 aligned indices, 16-entry
tables of four bits, four dimensions per Philox block): bit-exact against the CPU oracle, with
the words around the output untouched."""
import numpy as np
import pytest

from oracle import oracle as O

pytestmark = pytest.mark.gpu

KINDS = ["sobol", "sobol_owen", "niederreiter", "philox", "halton", "hammersley", "faure"]
# (dims, first, count): within a tile, up to and over its edges, several tiles, one dimension to all,
# the last indices of a 32-bit sequence
RANGES = [(1, 1, 1), (2, 255, 1), (3, 256, 256), (4, 255, 3), (5, 17, 239), (7, 17, 240), (8, 511, 1026),
          (33, 1, 300), (255, 250, 13), (256, 1023, 2), (4, 2 ** 32 - 300, 300)]


@pytest.fixture(scope="module")
def Q():
    from paper_2406_15632_gb300 import build as B
    from paper_2406_15632_gb300 import qmcrt

    B.build()
    qmcrt.load()
    return qmcrt


@pytest.mark.parametrize("dims,first,count", RANGES)
@pytest.mark.parametrize("fmt", ["u32", "f32", "f64"])
@pytest.mark.parametrize("kind", KINDS)
def test_points_at_tile_edges(Q, kind, fmt, dims, first, count):
    import torch

    if fmt == "u32" and kind in ("halton", "hammersley", "faure"):
        pytest.skip("no integer form")
    total = first + count - 1 if kind == "hammersley" else 0
    dt = {"u32": torch.int32, "f32": torch.float32, "f64": torch.float64}[fmt]
    for shift in (0, 1):  # an output that does not start on 16 bytes
        buf = torch.full((count * dims + 8,), -7, dtype=dt, device="cuda")
        out = buf[shift:shift + count * dims]
        Q.generate_points(kind, dims, first, count, fmt, seed=77, total_n=total, out=out)
        torch.cuda.synchronize()
        got = out.cpu().numpy().reshape(count, dims)
        ref = O.generate_points(kind, dims, first, count, fmt, seed=77, total_n=total)
        assert np.array_equal(got.view(np.uint8), ref.view(np.uint8))
        assert bool((buf[:shift] == -7).all()) and bool((buf[shift + count * dims:] == -7).all())

"""Padded copies of grids of short, single-cell and long odd rows, several rounds of the kernel's
blocks long, against numpy."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("pad", [8, 9])
@pytest.mark.parametrize("shape", [(20_000, 1, 1), (1, 20_000, 4), (1, 1, 20_000), (1, 1, 1), (3, 700, 1), (160, 171, 203),
                                   (180, 190, 200)])
def test_padded_copy(shape, pad):
    import torch

    from paper_2406_15632_gb300 import build as B
    from paper_2406_15632_gb300 import qmcrt as Q

    B.build()
    Q.load()
    g = np.random.default_rng(1).uniform(-0.2, 1.0, size=shape).astype(np.float32)
    g.flat[0] = np.nan
    ref = np.full([n + 2 * pad for n in shape], -0.0, dtype=np.float32)
    ref[pad:-pad, pad:-pad, pad:-pad] = np.where(g > 0, g, 0.0)
    src = torch.from_numpy(g).cuda()
    dst = torch.full((ref.size + 8,), 5.0, device="cuda")
    Q.qmcrt_pad_grid(src.data_ptr(), shape[2], shape[1], shape[0], pad, dst.data_ptr())
    torch.cuda.synchronize()
    out = dst.cpu().numpy()
    assert np.array_equal(out[:ref.size].view(np.uint32), ref.ravel().view(np.uint32))
    assert (out[ref.size:] == 5.0).all()

"""Direct light of a star that fills an image of more than 2^32 pixels: the last rows lie beyond a
32-bit pixel index, and equal the first ones by symmetry."""
import pytest

from paper_2406_15632_gb300 import scenes as S

pytestmark = pytest.mark.gpu

NX, NY, ROWS = 1 << 16, (1 << 16) + 8, 8


def test_last_rows_mirror_the_first():
    import numpy as np
    import torch

    from paper_2406_15632_gb300 import build as B
    from paper_2406_15632_gb300 import qmcrt as Q

    B.build()
    Q.load()
    if torch.cuda.mem_get_info()[0] < 24 * NX * NY + (8 << 30):
        pytest.skip("not enough device memory")
    p = S.Problem(grid=np.zeros((2, 2, 2), np.float32), lo=(-2.0,) * 3, hi=(2.0,) * 3, source="sphere", star_r=1.0,
                  limb_u=0.6, half_width=0.5, nx=NX, ny=NY)
    sc = Q.Scene(p, sky=0, tail=False)
    a = sc.accum_buffer("i64")
    sc.direct_light(a, subsamples=1, frac_bits=60)
    torch.cuda.synchronize()
    img = a.view(3, NY, NX)[0]
    first, last = img[:ROWS].double(), img[-ROWS:].flip(0).double()
    assert bool((last > 0).all())
    # sky points and brightness to a few float roundings
    assert bool(((first - last).abs() <= 1e-4 * first).all())
    del a, img, first, last
    torch.cuda.empty_cache()

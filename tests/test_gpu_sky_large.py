"""Bound map of a grid of more than 2^32 cells: the upper layers lie beyond a 32-bit index."""
import pytest

pytestmark = pytest.mark.gpu

N, TOP, M = 1632, 1612, 4096  # (N + 2)^3 = 4.36e9 cells; dense from layer TOP on


def test_bound_beyond_32_bit_indices():
    import torch

    from paper_2406_15632_gb300 import build as B
    from paper_2406_15632_gb300 import qmcrt as Q

    B.build()
    Q.load()
    lo, hi = (-1.0,) * 3, (1.0,) * 3
    need = Q.qmcrt_sky_workspace_bytes(N, N, N, lo, hi, 0.0)
    if torch.cuda.mem_get_info()[0] < 4 * N ** 3 + need + (8 << 30):
        pytest.skip("not enough device memory")
    g = torch.zeros((N, N, N), device="cuda")
    g[TOP:] = 1.0
    ws = torch.empty(need // 8 + 32, dtype=torch.float64, device="cuda")
    sky = torch.empty((6, M, M), dtype=torch.float64, device="cuda")
    Q.qmcrt_sky_bound(g.data_ptr(), N, N, N, lo, hi, 0.0, M, sky.data_ptr(), ws.data_ptr(), need,
                      torch.cuda.current_stream().cuda_stream)
    torch.cuda.synchronize()
    up, down = sky[4], sky[5]  # +z, -z
    assert bool(torch.isfinite(up).all())
    # depth of the texels' centre rays: layers TOP to N, along 1 / cos
    c = (torch.arange(M, device="cuda", dtype=torch.float64) + 0.5) * (2.0 / M) - 1.0
    depth = (N - TOP) * (2.0 / N) * torch.sqrt(1.0 + c[:, None] ** 2 + c[None, :] ** 2)
    inner = (c[:, None].abs() < 0.99) & (c[None, :].abs() < 0.99)  # rays that leave through the top face
    assert bool((up[inner] >= depth[inner]).all())
    # the neighbourhoods add two layers at most
    assert bool((up[inner] <= depth[inner] * (1.001 + 2.0 / (N - TOP))).all())
    assert bool((down == 0.0).all())
    del g, ws, sky, up, down
    torch.cuda.empty_cache()

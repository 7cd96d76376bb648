"""Gradient of the learned warp at the edges of its tiles: single rows, one row short of and past
a 128-row tile, fewer and more tiles than CTAs, rows of weight zero, gradients that do not start
on 16 bytes and that hold something already.  Against the oracle with bf16 weights, features,
activations and backward signals; where float sums round to the other neighbour a signal
differs by one bf16 step, 2^-8 of it, which bounds the relative difference."""
import numpy as np
import pytest

from oracle import flow as F

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def Q():
    from paper_2406_15632_gb300 import build as B
    from paper_2406_15632_gb300 import qmcrt

    B.build()
    qmcrt.load()
    return qmcrt


@pytest.mark.parametrize("n", [1, 5, 127, 128, 129, 300, 128 * 76, 128 * 76 + 1, 128 * 160 + 3])
@pytest.mark.parametrize("mix", [0.0, 0.1])
def test_gradient_at_tile_edges(Q, n, mix):
    import torch

    vec = F.init_params(n % 7, scale=1.5)
    W = Q.Warp(vec, rows=128, uniform_mix=mix)
    rng = np.random.default_rng(n)
    x = rng.uniform(size=(n, 3)).astype(np.float32)
    x[rng.uniform(size=(n, 3)) < 0.02] = 1.0  # the upper end of the last bin
    w = rng.lognormal(size=n).astype(np.float32)
    if n > 4:
        w[::3] = 0.0
    lr, gr = F.loss_and_grad(x.astype(np.float64), w.astype(np.float64), vec, use_bf16=True, mix=mix)
    xd, wd = torch.tensor(x).cuda(), torch.tensor(w).cuda()
    for shift in (0, 1):
        buf = torch.full((Q.WARP_PARAMS + 4,), 0.5, device="cuda")
        loss = torch.full((1,), 2.0, device="cuda")
        Q.qmcrt_warp_grad(W.desc, xd.data_ptr(), wd.data_ptr(), n, buf.data_ptr() + 4 * shift, loss.data_ptr(),
                          W.ws.data_ptr(), W.ws_bytes, torch.cuda.current_stream().cuda_stream)
        torch.cuda.synchronize()
        assert W.error.item() == 0
        got = buf.cpu().numpy().astype(np.float64)
        assert (got[:shift] == 0.5).all() and (got[shift + Q.WARP_PARAMS:] == 0.5).all()
        g = got[shift:shift + Q.WARP_PARAMS] - 0.5
        # adding to 0.5 rounds each value to 2^-25 several times over
        slack = 64 * 2.0 ** -25 * np.sqrt(Q.WARP_PARAMS)
        assert np.linalg.norm(g - gr) <= 2.0 ** -8 * np.linalg.norm(gr) + slack
        assert loss.item() - 2.0 == pytest.approx(lr, rel=1e-4, abs=1e-5)

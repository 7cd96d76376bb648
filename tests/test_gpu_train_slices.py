"""Gradient of the learned warp over slices of several tiles: weight gradients that accumulate over
the tiles of a slice, slices that end within a tile, several slices a pass and several passes.
Against the oracle with bf16 weights, features, activations and backward signals, within one bf16
step (2^-8) of it, as float sums that round to the other neighbour differ."""
import numpy as np
import pytest

from oracle import flow as F

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("rows,n", [(1152, 577), (1152, 1151), (1152, 1152), (1152, 1153), (1152, 2 * 1152 + 577),
                                    (1 << 14, 10_000), (1 << 14, (1 << 14) + 4097), (1 << 16, 40_001)])
def test_gradient_over_slices(rows, n):
    import torch

    from paper_2406_15632_gb300 import build as B
    from paper_2406_15632_gb300 import qmcrt as Q

    B.build()
    Q.load()
    vec = F.init_params(n % 5, scale=1.5)
    W = Q.Warp(vec, rows=rows, uniform_mix=0.1)
    rng = np.random.default_rng(n)
    x = rng.uniform(size=(n, 3)).astype(np.float32)
    w = rng.lognormal(size=n).astype(np.float32)
    lr, gr = F.loss_and_grad(x.astype(np.float64), w.astype(np.float64), vec, use_bf16=True, mix=0.1)
    xd, wd = torch.tensor(x).cuda(), torch.tensor(w).cuda()
    g = torch.zeros(Q.WARP_PARAMS, device="cuda")
    loss = torch.zeros(1, device="cuda")
    Q.qmcrt_warp_grad(W.desc, xd.data_ptr(), wd.data_ptr(), n, g.data_ptr(), loss.data_ptr(), W.ws.data_ptr(), W.ws_bytes,
                      torch.cuda.current_stream().cuda_stream)
    torch.cuda.synchronize()
    assert W.error.item() == 0
    d = g.cpu().numpy().astype(np.float64) - gr
    assert np.linalg.norm(d) <= 2.0 ** -8 * np.linalg.norm(gr)
    # every matrix and bias for itself: a slice or tile left out or taken twice is a share of it
    bounds = np.cumsum([0, 32] + [s for _ in range(2) for l in range(4) for s in ((32 if l == 3 else 128) * 128,
                                                                                 32 if l == 3 else 128)])
    assert bounds[-1] == Q.WARP_PARAMS
    for a, b in zip(bounds[:-1], bounds[1:]):
        assert np.linalg.norm(d[a:b]) <= 2.0 ** -7 * np.linalg.norm(gr[a:b])
    assert loss.item() == pytest.approx(lr, rel=1e-4, abs=1e-5)

"""The wavefront's regrouping at the edges of its bucket counts: workspaces whose queues hold
fewer cursors than the key has buckets, queues that fill few buckets, and chunks on both
sides of the size at which the key grows.  Images equal the one-kernel tracer's bit for bit."""
import pytest

from paper_2406_15632_gb300 import scenes as S

pytestmark = pytest.mark.gpu

PROB = S.clumpy_problem(n=16, max_orders=5, nx=24, ny=20, per_order=True)


@pytest.fixture(scope="module")
def Q():
    from paper_2406_15632_gb300 import build as B
    from paper_2406_15632_gb300 import qmcrt

    B.build()
    qmcrt.load()
    return qmcrt


@pytest.mark.parametrize("precision,ws_packets,first,count", [
    ("f32", 1, 5, 3), ("f32", 2, 1, 9), ("f64", 1, 2, 3), ("f32", 64, 33, 200), ("f32", 1 << 12, 1, 1),
    ("f32", 1 << 12, 77, 4000), ("f64", 1 << 12, 77, 4000), ("f32", 1 << 20, 3, (1 << 20) - 5),
    ("f32", 1 << 21, 1 << 21, 1 << 21), ("f32", 1 << 21, 9, (1 << 21) + 4097)])
def test_regrouping_keeps_the_images(Q, precision, ws_packets, first, count):
    import torch

    sc = Q.Scene(PROB)
    a, b = sc.accum_buffer("i64"), sc.accum_buffer("i64")
    sc.trace(first, count, a, frac_bits=32, precision=precision)
    ws = sc.wavefront_workspace(ws_packets, precision)
    for _ in range(2):  # the second run finds the first one's queues and counters in the workspace
        b.zero_()
        sc.trace_wavefront(first, count, b, ws, frac_bits=32, precision=precision)
    torch.cuda.synchronize()
    assert torch.equal(a, b)
    assert bool((a != 0).any())

"""Timed cases of the library: the calls a program makes through the package's public entry
points, over the range of sizes and options it is used at.

A case is a dict of plain values.  prepare() makes what a program holds before the call (the
density grid on the device, the scene with its maps, buffers, a trained proposal), run() is
one pass, exact() is the same result from plain torch in 64 bits.  Every input follows from
the seed: the medium's parameters, the viewing angle, the dust, the range of point indices
and the scrambling or Philox key.
"""
from __future__ import annotations

import math
import random

import torch

from paper_2406_15632_gb300 import qmcrt as Q
from paper_2406_15632_gb300 import scenes as S

# Cells a packet must cross per cell of the grid's edge (tau_1 walk of the rays that can
# scatter, peel-off walk while the depth left ahead can matter); the repository counts 155.7
# per packet on the 256^3 disk and 2566 over the 20 orders of the 128^3 clumpy envelope.
CELLS_PER_EDGE = {"disk": 0.61, "shell": 1.0, "clumpy": 1.0}
OPS_PER_CELL, OPS_PER_PACKET = 10.0, 150.0  # cell step; emission, phase function, projection
WARP_WEIGHTS = 2 * (3 * 128 * 128 + 32 * 128)


def listed() -> list[dict]:
    return [
        # the smallest render: a look at a coarse model, where launches and latency count
        dict(name="disk_smallest", kind="single", medium="disk", n=32, count=4096, px=64, generator="sobol",
             splat="nearest", source="point", precision="f32"),
        # an interactive preview: odd sizes, a ragged packet range, scrambled points, tent splat
        dict(name="disk_preview", kind="single", medium="disk", n=100, count=1_000_003, px=200,
             generator="sobol_owen", splat="bilinear", source="point", precision="f32"),
        # the headline workload: one step of the 256^3 disk, the largest single launch
        dict(name="disk_headline", kind="single", medium="disk", n=256, count=1 << 26, px=256, generator="sobol",
             splat="nearest", source="point", precision="f32"),
        # a reference-grade image: FP64, a finite star, Halton points (the comparison of sequences)
        dict(name="star_reference_f64", kind="single", medium="disk", n=64, count=200_000, px=100,
             generator="halton", splat="nearest", source="sphere", precision="f64"),
        # one trace feeding eight viewing angles (inclinations from the pole to the edge)
        dict(name="observers_8", kind="observers", medium="disk", n=256, count=1 << 22, px=256, observers=8,
             generator="sobol", splat="nearest", source="point", precision="f32"),
        # multiple scattering of a small problem in one kernel, an image per order, plain Monte Carlo
        dict(name="orders_small", kind="multiple", medium="clumpy", n=32, count=30_000, px=64, orders=8,
             per_order=True, generator="philox", splat="nearest", source="point", precision="f32"),
        # the multiple-scattering workload: 20 orders of the clumpy envelope as a wavefront
        dict(name="clumpy_wavefront", kind="wavefront", medium="clumpy", n=128, count=1 << 22, px=512, orders=20,
             per_order=False, generator="sobol", splat="nearest", source="point", precision="f32"),
        # a short learned render: points, warp on the tensor cores, wavefront trace, FP64 image
        dict(name="learned_render", kind="learned", medium="clumpy", n=128, count=1 << 18, px=512, orders=20,
             per_order=False, generator="sobol_owen", splat="nearest", source="point", precision="f32"),
        # one optimiser step of the proposal's training: forward, backward, Adam on a minibatch
        dict(name="train_step", kind="train", rows=1 << 16),
        # many problems in one graph replay: instances of the finite-star disk
        dict(name="batch_24", kind="batch", medium="disk", n=256, instances=24, min_log2=18, max_log2=22, px=256,
             generator="sobol", splat="nearest", source="sphere", precision="f32"),
        # end to end from host memory: a new grid in, maps rebuilt, trace, image out
        dict(name="host_render", kind="host", medium="disk", n=256, count=1 << 22, px=256, generator="sobol",
             splat="nearest", source="point", precision="f32"),
        # the point sets themselves: all coordinates of the 20-order workload
        dict(name="points_80", kind="points", count=1 << 20, dims=80, generator="sobol", fmt="f32"),
    ]


def _log_int(rng: random.Random, lo: int, hi: int) -> int:
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _count(rng: random.Random, lo: int, hi: int) -> int:
    """A packet count, every other one a power of two (aligned blocks of a sequence)."""
    c = _log_int(rng, lo, hi)
    return 1 << (c.bit_length() - 1) if rng.random() < 0.5 else c


def draw(rng: random.Random) -> dict:
    kind = rng.choice(["single", "single", "single", "observers", "multiple", "wavefront", "wavefront", "learned",
                       "train", "batch", "host", "points"])
    generator = rng.choice(["sobol", "sobol", "sobol_owen", "halton", "philox"])
    if kind == "train":
        return dict(kind=kind, rows=_log_int(rng, 1 << 9, 1 << 17))
    if kind == "points":
        dims = _log_int(rng, 2, 120)
        return dict(kind=kind, dims=dims, count=_log_int(rng, 1 << 9, (1 << 26) // dims), generator=generator,
                    fmt=rng.choice(["f32", "f32", "f64", "u32"]) if generator != "halton" else
                    rng.choice(["f32", "f64"]))
    c = dict(kind=kind, px=_log_int(rng, 32, 512), splat=rng.choice(["nearest", "nearest", "bilinear"]),
             generator=generator, source=rng.choice(["point", "point", "sphere"]), precision="f32")
    if kind in ("multiple", "wavefront", "learned"):
        c.update(medium=rng.choice(["clumpy", "clumpy", "disk"]), n=_log_int(rng, 24, 128),
                 orders=rng.randint(2, 20), per_order=rng.random() < 0.3)
        hi = {"multiple": 1 << 18, "wavefront": 1 << 21, "learned": 1 << 20}[kind]
        c["count"] = _count(rng, 1 << 10, hi)
        if kind == "learned":  # the proposal warps a point source's first order
            c.update(source="point", generator=rng.choice(["sobol", "sobol_owen"]))
        elif c["count"] <= 1 << 16 and rng.random() < 0.2:
            c["precision"] = "f64"
        return c
    c.update(medium=rng.choice(["disk", "disk", "shell", "clumpy"]), n=_log_int(rng, 24, 256))
    if kind == "batch":
        lo = rng.randint(10, 16)
        c.update(source="sphere", instances=_log_int(rng, 2, 40), min_log2=lo, max_log2=lo + rng.randint(1, 4),
                 generator=rng.choice(["sobol", "sobol_owen"]))
    elif kind == "observers":
        c.update(observers=rng.randint(2, 16), count=_count(rng, 1 << 10, 1 << 21))
    elif kind == "host":
        c["count"] = _count(rng, 1 << 12, 1 << 23)
    else:
        c["count"] = _count(rng, 1 << 10, 1 << 24)
        if c["count"] <= 1 << 19 and rng.random() < 0.3:
            c["precision"] = "f64"
    return c


# --- inputs ---------------------------------------------------------------------------------

def _centres(n: int) -> torch.Tensor:
    return -1.0 + (torch.arange(n, dtype=torch.float64, device="cuda") + 0.5) * (2.0 / n)


def _grid(case: dict, seed: int) -> torch.Tensor:
    """The density grid [n][n][n] (kappa rho, FP32): the shapes of the package's scenes, with
    parameters that follow from the seed."""
    n, r = case["n"], random.Random(seed)
    c = _centres(n)
    z, y, x = c[:, None, None], c[None, :, None], c[None, None, :]
    if case["medium"] == "disk":  # flared disk: r^-alpha exp(-z^2 / 2 h^2), h = h0 r^beta
        k0, h0 = r.uniform(0.8, 1.2) / 9.0, r.uniform(0.09, 0.11)
        rad = torch.sqrt(x * x + y * y).clamp_min(1e-9)
        k = k0 * rad ** -2.0 * torch.exp(-0.5 * (z / (h0 * rad ** 1.25)) ** 2)
        k = torch.where((rad >= 0.1) & (rad <= 1.0), k, 0.0)
    elif case["medium"] == "shell":  # thin dust shell
        rad = torch.sqrt(x * x + y * y + z * z)
        k = torch.where((rad >= 500 / 600) & (rad <= 550 / 600), r.uniform(0.05, 0.2) * 12.0, 0.0)
    else:  # clumpy envelope: r^-1.5 times a log-normal field smoothed over four cells, radial tau 5
        g = torch.Generator(device="cuda").manual_seed(seed)
        white = torch.randn((n, n, n), generator=g, device="cuda", dtype=torch.float64)
        f = torch.fft.fftfreq(n, device="cuda", dtype=torch.float64)
        f2 = f[:, None, None] ** 2 + f[None, :, None] ** 2 + f[None, None, :] ** 2
        G = torch.fft.ifftn(torch.fft.fftn(white) * torch.exp(-2.0 * (math.pi * 4.0) ** 2 * f2)).real
        G = (G - G.mean()) / G.std()
        rad = torch.sqrt(x * x + y * y + z * z).clamp_min(1e-9)
        k0 = 5.0 / ((1.0 - 0.05 ** -0.5) / -0.5)
        k = torch.where((rad >= 0.05) & (rad <= 1.0), k0 * rad ** -1.5 * torch.exp(G - 0.5), 0.0)
    return k.to(torch.float32).contiguous()


def _problem(case: dict, seed: int, grid) -> S.Problem:
    r = random.Random(seed + 1)
    star = dict(source="sphere", star_r=0.05, limb_u=0.6) if case["source"] == "sphere" else {}
    multi = {}
    if "orders" in case:
        multi = dict(max_orders=case["orders"], per_order=case["per_order"], rr_threshold=1e-4, rr_survival=0.1)
    return S.Problem(grid=grid, albedo=r.uniform(0.55, 0.75), g=r.uniform(0.4, 0.6), p_l=0.5,
                     theta_obs=math.pi / 4 + r.uniform(-0.2, 0.2), half_width=1.0, nx=case["px"], ny=case["px"],
                     splat=case["splat"], generator=case["generator"], seed=r.randrange(1 << 31), **star, **multi)


def _first(case: dict, seed: int) -> int:
    """First point index: an aligned block for a power of two, anywhere else otherwise."""
    r, n = random.Random(seed + 2), case["count"]
    return n * r.randint(1, 7) if n & (n - 1) == 0 else r.randint(1, 1 << 20)


def _angles(case: dict, seed: int) -> list[tuple[float, float]]:
    phi, m = random.Random(seed + 3).uniform(0.0, 0.5), case["observers"]
    return [(math.radians(90.0 * k / (m - 1)), phi) for k in range(m)]


def _instances(case: dict, seed: int) -> list[S.Instance]:
    """Inclinations x wavelengths with budgets spread over the case's range (the package's
    batched workload, cut to the case's number of instances)."""
    r, m, span = random.Random(seed + 4), case["instances"], case["max_log2"] - case["min_log2"] + 1
    budgets = [1 << (case["min_log2"] + j % span) for j in range(m)]  # one total whatever the seed
    r.shuffle(budgets)
    out = []
    for j, n in enumerate(budgets):
        t = r.random()
        out.append(S.Instance(theta_obs=math.radians(90.0 * (j // 4) / max(1, (m - 1) // 4)), albedo=0.4 + 0.5 * t,
                              g=0.2 + 0.5 * t, kscale=0.5 * 8.0 ** t, n_packets=n, first_index=n))
    return out


def _warp_params(seed: int) -> torch.Tensor:
    """A proposal as training leaves it: output layers and the first density well off uniform."""
    p = Q.Warp.initial(seed)
    r = torch.Generator().manual_seed(seed + 5)
    p[:32] = 0.5 * torch.randn(32, generator=r)
    for m in range(2):
        o = 32 + m * (WARP_WEIGHTS // 2 + 3 * 128 + 32) + 3 * (128 * 128 + 128)
        p[o:o + 32 * 128] *= 5.0
    return p


def _training_data(case: dict, seed: int):
    """Logged samples: coordinates crowded toward one end, weights over a few decades."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    x = torch.rand((case["rows"], 3), generator=g, device="cuda") ** torch.tensor([1.0, 1.5, 2.0], device="cuda")
    w = torch.exp(1.5 * torch.randn(case["rows"], generator=g, device="cuda"))
    return x, w


def _moments(seed: int):
    """Adam moments in the middle of a training."""
    g = torch.Generator(device="cuda").manual_seed(seed + 6)
    m = 1e-4 * torch.randn(Q.WARP_PARAMS, generator=g, device="cuda")
    v = 1e-6 * (0.5 + torch.rand(Q.WARP_PARAMS, generator=g, device="cuda"))
    return m, v


ADAM_STEP, ADAM_LR, MIX = 100, 2e-3, 0.1


def prepare(case: dict, seed: int) -> dict:
    kind = case["kind"]
    if kind == "points":
        return dict(case=case, first=random.Random(seed).randint(1, 1 << 24), seed=seed)
    if kind == "train":
        x, w = _training_data(case, seed)
        warp = Q.Warp(_warp_params(seed), rows=case["rows"], uniform_mix=MIX)
        m, v = _moments(seed)
        warp.m.copy_(m)
        warp.v.copy_(v)
        warp.step = ADAM_STEP
        return dict(case=case, warp=warp, x=x, w=w)
    grid = _grid(case, seed)
    if kind == "host":
        host = torch.empty(grid.shape, dtype=torch.float32, pin_memory=True)
        host.copy_(grid)
        prob = _problem(case, seed, host)
        image = torch.empty((1, 3, prob.ny, prob.nx), dtype=torch.float64, pin_memory=True)
        return dict(case=case, renderer=Q.HostRenderer(prob, case["count"], precision=case["precision"]), host=host,
                    image=image, first=_first(case, seed))
    prob = _problem(case, seed, grid)
    sc = Q.Scene(prob, grid_device=grid)
    if kind == "batch":
        b = Q.Batch(prob, _instances(case, seed), scene=sc, precision=case["precision"], chunk_log2=24,
                    packets_per_thread=1)
        b.capture()
        return dict(case=case, batch=b)
    st = dict(case=case, scene=sc, first=_first(case, seed), frac_bits=Q.default_frac_bits(prob, case["count"]))
    if kind == "observers":
        st["angles"] = _angles(case, seed)
        st["buf"] = torch.zeros((case["observers"], 1, 3, prob.ny, prob.nx), dtype=torch.int64, device="cuda")
        sc.observer_array(st["angles"])  # the tail maps of the angles, kept by the scene
    elif kind == "learned":
        warp = Q.Warp(_warp_params(seed), rows=1 << 12, uniform_mix=MIX)
        st["tracer"] = Q.LearnedTracer(sc, warp, chunk=1 << 20, wavefront=True, precision=case["precision"])
        st["buf"] = sc.accum_buffer("f64")
    else:
        st["buf"] = sc.accum_buffer("i64")
        if kind == "wavefront":
            st["ws"] = sc.wavefront_workspace(case["count"], case["precision"])
    return st


def run(st: dict):
    case = st["case"]
    kind = case["kind"]
    if kind == "points":
        return Q.generate_points(case["generator"], case["dims"], st["first"], case["count"], case["fmt"],
                                 seed=st["seed"])
    if kind == "train":
        warp = st["warp"]
        loss, grad = warp.gradient(st["x"], st["w"])
        warp.adam_step(lr=ADAM_LR)
        return [loss, grad, warp.params, warp.m, warp.v]
    if kind == "batch":
        st["batch"].replay()
        return st["batch"].out
    if kind == "host":
        st["renderer"](st["host"], st["first"], case["count"], st["image"])
        return st["image"]
    sc, buf, fb = st["scene"], st["buf"], st["frac_bits"]
    first, count, prec = st["first"], case["count"], case["precision"]
    buf.zero_()
    if kind == "learned":
        st["tracer"].trace(first, count, buf, accum="f64", precision=prec)
        return sc.reduce(buf, 1.0 / count, accum="f64")
    if kind == "observers":
        sc.trace_observers(st["angles"], first, count, buf, frac_bits=fb, precision=prec)
        return [sc.reduce(buf[o], 1.0 / count, frac_bits=fb) for o in range(case["observers"])]
    if kind == "wavefront":
        sc.trace_wavefront(first, count, buf, st["ws"], frac_bits=fb, precision=prec)
    else:
        sc.trace(first, count, buf, frac_bits=fb, precision=prec)
    return sc.reduce(buf, 1.0 / count, frac_bits=fb)


def work(case: dict) -> dict:
    kind = case["kind"]
    if kind == "points":
        size = 8 if case["fmt"] == "f64" else 4
        # one XOR and one select per bit of the index (the digits of a radical inverse alike)
        return dict(bytes=float(size * case["count"] * case["dims"]), flops=64.0 * case["count"] * case["dims"])
    if kind == "train":  # forward and the two backward products; samples in, state in and out
        return dict(bytes=16.0 * case["rows"] + 4.0 * 107360 * 7, flops=6.0 * WARP_WEIGHTS * case["rows"])
    n, px = case["n"], case["px"]
    images, packets, walks = 1, case.get("count", 0), 1.0
    if kind == "batch":
        images, packets = case["instances"], sum(i.n_packets for i in _instances(case, 0))
    elif kind == "observers":
        images, walks = case["observers"], 0.5 + 0.5 * case["observers"]
    elif "orders" in case:
        images = case["orders"] if case["per_order"] else 1
        walks = float(case["orders"])
    cells = CELLS_PER_EDGE[case["medium"]] * n * walks
    flops = packets * (cells * OPS_PER_CELL + OPS_PER_PACKET * walks)
    if kind == "learned":
        flops += 2.0 * WARP_WEIGHTS * packets
    return dict(bytes=4.0 * n ** 3 + 24.0 * px * px * images, flops=flops)


# --- the same results in 64 bits ---------------------------------------------------------------
# Plain torch: the points, then all packets of a chunk together through emission, the cell
# walk, forced scattering, peel-off toward the observer and binning.

MASK32 = 0xFFFFFFFF


def _fmix32(h):
    h = h ^ (h >> 16)
    h = (h * 0x85EBCA6B) & MASK32
    h = h ^ (h >> 13)
    h = (h * 0xC2B2AE35) & MASK32
    return h ^ (h >> 16)


def _brev(x: torch.Tensor) -> torch.Tensor:
    for s, m in ((1, 0x55555555), (2, 0x33333333), (4, 0x0F0F0F0F), (8, 0x00FF00FF), (16, 0x0000FFFF)):
        x = ((x >> s) & m) | ((x & m) << s)
    return x


def _primes(n: int) -> list[int]:
    out, c = [], 2
    while len(out) < n:
        if all(c % p for p in out):
            out.append(c)
        c += 1
    return out


class _Points:
    """Coordinates of point indices, dimension by dimension: 32-bit integers (bits) or values."""

    def __init__(self, generator: str, dims: int, seed: int, device):
        self.generator, self.seed = generator, seed
        self.primes = _primes(dims)
        if generator.startswith("sobol"):  # torch's direction numbers, left-aligned in 30 bits
            self.v = torch.quasirandom.SobolEngine(dims).sobolstate.tolist()
        self.device = device

    def bits(self, i: torch.Tensor, d: int) -> torch.Tensor:
        if self.generator == "philox":
            return self._philox(i, d)
        g, x = i ^ (i >> 1), torch.zeros_like(i)
        for k in range(30):  # indices below 2^30
            x ^= ((g >> k) & 1) * (self.v[d][k] << 2)
        if self.generator == "sobol_owen":
            s = _fmix32((self.seed & MASK32) ^ _fmix32(((self.seed >> 32) + 0x9E3779B9 * (d + 1)) & MASK32))
            r = (_brev(x) + s) & MASK32
            for c in (0x6A09E666, 0xBB67AE84, 0x3C6EF372, 0xA54FF53A):
                r = r ^ ((r * c) & MASK32)
            x = _brev(r)
        return x

    def _philox(self, i, d):
        c = [i & MASK32, (i >> 32) & MASK32, torch.full_like(i, d >> 2), torch.zeros_like(i)]
        k0, k1 = self.seed & MASK32, (self.seed >> 32) & MASK32
        for r in range(10):
            if r:
                k0, k1 = (k0 + 0x9E3779B9) & MASK32, (k1 + 0xBB67AE85) & MASK32
            p0, p1 = c[0] * 0xD2511F53, c[2] * 0xCD9E8D57  # 64-bit products, modulo 2^64
            c = [((p1 >> 32) & MASK32) ^ c[1] ^ k0, p1 & MASK32, ((p0 >> 32) & MASK32) ^ c[3] ^ k1, p0 & MASK32]
        return c[d & 3]

    def __call__(self, i: torch.Tensor, d: int) -> torch.Tensor:
        if self.generator != "halton":
            return self.bits(i, d).double() * 2.0 ** -32
        b, num, den = self.primes[d], torch.zeros_like(i), torch.ones_like(i)
        while bool((i > 0).any()):
            more = i > 0
            num = torch.where(more, num * b + i % b, num)
            den = torch.where(more, den * b, den)
            i = i // b
        return num.double() / den.double()


def _sincos2pi(u):
    """sin and cos of 2 pi u, exact at quarter turns."""
    k = torch.round(4.0 * u)
    f = (u - 0.25 * k) * (2.0 * math.pi)
    s, c, q = torch.sin(f), torch.cos(f), k.long() % 4
    sn = torch.where(q == 0, s, torch.where(q == 1, c, torch.where(q == 2, -s, -c)))
    cs = torch.where(q == 0, c, torch.where(q == 1, -s, torch.where(q == 2, -c, s)))
    return sn, cs


def _dot(a, b):
    return (a * b).sum(-1)


def _unit(a):
    return a / a.norm(dim=-1, keepdim=True)


def _walk(grid, p, d, target=None):
    """Optical depth (raw cell values) from p along d through [-1, 1]^3 to the edge; with a
    target, also the path length at which it is reached (the end of the last cell of nonzero
    density where it is not)."""
    n, dev, N = grid.shape[0], grid.device, p.shape[0]
    flat, h = grid.reshape(-1).double(), 2.0 / grid.shape[0]
    stride = torch.tensor([1, n, n * n], device=dev)
    c = torch.floor((p + 1.0) / h)
    c = torch.where(p < -1.0 + c * h, c - 1, torch.where(p >= -1.0 + (c + 1) * h, c + 1, c))
    c = torch.where((d < 0) & (p == -1.0 + c * h), c - 1, c)
    nxt = torch.where(d != 0, (-1.0 + (c + (d > 0)) * h - p) / d, math.inf)
    cell, step = c.long(), torch.sign(d).long()
    dt = torch.where(d != 0, h / d.abs(), 0.0)
    tau, t_hit = torch.zeros(N, device=dev, dtype=torch.float64), torch.zeros(N, device=dev, dtype=torch.float64)
    inside = ((cell >= 0) & (cell < n)).all(1)
    live = torch.nonzero(inside).squeeze(1)
    cell, step, nxt, dt = cell[live], step[live], nxt[live], dt[live]
    t, acc, last = (torch.zeros(len(live), device=dev, dtype=torch.float64) for _ in range(3))
    goal = None if target is None else target[live]
    on = torch.ones(len(live), device=dev, dtype=torch.bool)
    steps = 0
    while len(live):
        t1, ax = nxt.min(1)
        k = flat[(cell * stride).sum(1)]
        add = torch.where(on, k * (t1 - t), 0.0)
        if target is not None:
            hit = on & (k > 0) & (acc + add >= goal)
            last = torch.where(hit, t + (goal - acc) / k, torch.where(on & (add > 0), t1, last))
            on = on & ~hit
        acc, t = acc + add, t1
        ax = ax[:, None]
        cell.scatter_add_(1, ax, step.gather(1, ax))
        nxt.scatter_add_(1, ax, dt.gather(1, ax))
        c = cell.gather(1, ax).squeeze(1)
        on = on & (c >= 0) & (c < n)
        cell.clamp_(0, n - 1)
        steps += 1
        if steps % 8 == 0:  # retire finished rays
            off = ~on
            tau[live[off]], t_hit[live[off]] = acc[off], last[off]
            live, cell, step, nxt, dt = live[on], cell[on], step[on], nxt[on], dt[on]
            t, acc, last = t[on], acc[on], last[on]
            goal = None if goal is None else goal[on]
            on = on[on]
    return tau, t_hit


class _Tracer:
    def __init__(self, prob: S.Problem, grid: torch.Tensor):
        self.p, self.grid, self.dev = prob, grid, grid.device
        self.points = _Points(prob.generator, prob.dims, prob.seed, grid.device)

    def view(self, theta, phi):
        st, ct, sp, cp = math.sin(theta), math.cos(theta), math.sin(phi), math.cos(phi)
        v = lambda *a: torch.tensor(a, device=self.dev, dtype=torch.float64)
        return v(st * cp, st * sp, ct), v(-sp, cp, 0.0), v(-ct * cp, -ct * sp, st)

    def emit(self, i):
        p, u = self.p, self.points
        s, c = _sincos2pi(u(i, 0))
        v = u(i, 1)
        ct, st = 2.0 * v - 1.0, 2.0 * torch.sqrt((v * (1.0 - v)).clamp_min(0.0))
        n = torch.stack([st * c, st * s, ct], 1)
        a = torch.stack([ct * c, ct * s, -st], 1)
        if p.source == "point":
            return torch.zeros_like(n), n, a, torch.ones_like(ct), u(i, 2)
        e0 = 4 * p.max_orders if p.max_orders > 1 else 3  # the emission point across the direction
        q = u(i, e0)
        sp, cp = _sincos2pi(u(i, e0 + 1))
        mu = torch.sqrt((1.0 - q).clamp_min(0.0))
        b = torch.stack([-s, c, torch.zeros_like(s)], 1)
        pos = p.star_r * (torch.sqrt(q)[:, None] * (cp[:, None] * a + sp[:, None] * b) + mu[:, None] * n)
        return pos, n, a, (1.0 - p.limb_u + p.limb_u * mu) / (1.0 - p.limb_u / 3.0), u(i, 2)

    def peel(self, image, view, pos, n, a, St, kscale):
        """Add the peel-off of packets (Stokes St in the frame of axis a) to image [3][ny][nx]."""
        p = self.p
        k, ex, ey = view
        x, y = pos @ ex, pos @ ey
        seen = torch.ones_like(x, dtype=torch.bool)
        if p.source == "sphere":
            b, c = pos @ k, _dot(pos, pos) - p.star_r ** 2
            seen = ~((c <= 0) | ((b < 0) & (b * b - c > 0)))
        x, y, pos, n, a, St = x[seen], y[seen], pos[seen], n[seen], a[seen], St[seen]
        if not len(x):
            return
        kk = k.expand_as(pos)
        tau = _walk(self.grid, pos, kk)[0] * kscale
        mu = n @ k
        hg = (1.0 - p.g ** 2) / (1.0 + p.g ** 2 - 2.0 * p.g * mu) ** 1.5
        f = torch.exp(-tau) * hg / (4.0 * math.pi)
        r12 = -p.p_l * (1.0 - mu * mu) / (1.0 + mu * mu)
        r33 = 2.0 * mu / (1.0 + mu * mu)
        b = torch.linalg.cross(n, a)
        m = torch.linalg.cross(n, kk)
        m = torch.where(_dot(m, m)[:, None] < 1e-24, b, m)
        m = _unit(m)
        pin = torch.linalg.cross(m, n)
        q, u = self.turn(_dot(a, pin), _dot(b, pin), St[:, 1], St[:, 2])
        I, q, u = f * (St[:, 0] + r12 * q), f * (r12 * St[:, 0] + q), f * r33 * u
        q, u = self.turn(-(m @ ex), m @ ey, q, u)
        out = torch.stack([I, q, u])
        hw, nx, ny = p.half_width, p.nx, p.ny
        fx, fy = (x + hw) * (nx / (2.0 * hw)), (y + hw) * (ny / (2.0 * hw))
        if p.splat == "nearest":
            spots = [(torch.floor(fx), torch.floor(fy), 1.0)]
        else:
            fx, fy = fx - 0.5, fy - 0.5
            x0, y0 = torch.floor(fx), torch.floor(fy)
            ax, ay = fx - x0, fy - y0
            spots = [(x0 + i, y0 + j, (ax if i else 1.0 - ax) * (ay if j else 1.0 - ay))
                     for j in range(2) for i in range(2)]
        for ix, iy, w in spots:
            ok = (ix >= 0) & (ix < nx) & (iy >= 0) & (iy < ny)
            e = (iy * nx + ix).long()[ok]
            image.reshape(3, -1).index_add_(1, e, (out * w)[:, ok])

    @staticmethod
    def turn(c, s, q, u):
        c2, s2 = c * c - s * s, 2.0 * c * s
        return q * c2 + u * s2, -q * s2 + u * c2

    def trace(self, first, count, views, kscale=1.0, chunk=1 << 21):
        """Raw image sums [len(views)][n_images][3][ny][nx] of packets first .. first + count - 1."""
        p = self.p
        images = torch.zeros((len(views), p.n_images, 3, p.ny, p.nx), device=self.dev, dtype=torch.float64)
        for c0 in range(0, count, chunk):
            i = first + torch.arange(c0, min(c0 + chunk, count), device=self.dev)
            pos, n, a, wgt, wd = self.emit(i)
            St = torch.zeros_like(n)
            St[:, 0] = wgt
            for order in range(1, p.max_orders + 1):
                base = 4 * (order - 1)
                if order > 1:
                    self.scatter(self.points(i, base), self.points(i, base + 1), n, a, St)
                    wd = self.points(i, base + 2)
                tau1 = _walk(self.grid, pos, n)[0] * kscale
                live = tau1 >= p.tau_min
                i, pos, n, a, St, wd, tau1 = (v[live] for v in (i, pos, n, a, St, wd, tau1))
                W = -torch.expm1(-tau1)
                t = _walk(self.grid, pos, n, -torch.log1p(-wd * W) / kscale)[1]
                pos = pos + t[:, None] * n
                St = St * (W * p.albedo)[:, None]
                for o, v in enumerate(views):
                    self.peel(images[o, order - 1 if p.per_order else 0], v, pos, n, a, St, kscale)
                if order == p.max_orders:
                    break
                low = St[:, 0] < p.rr_threshold
                stay = ~low | (self.points(i, base + 3) < p.rr_survival)
                St = torch.where(low[:, None], St / p.rr_survival, St)
                i, pos, n, a, St = (v[stay] for v in (i, pos, n, a, St))
                if not len(i):
                    break
        return images

    def scatter(self, u, v, n, a, St):
        p = self.p
        f = (1.0 - p.g ** 2) / (1.0 - p.g + 2.0 * p.g * v)
        ct = ((1.0 + p.g ** 2 - f * f) / (2.0 * p.g)).clamp(-1.0, 1.0)
        st = torch.sqrt(((1.0 - ct) * (1.0 + ct)).clamp_min(0.0))
        s, c = _sincos2pi(u)
        b = torch.linalg.cross(n, a)
        m = c[:, None] * b - s[:, None] * a
        n[:] = _unit(ct[:, None] * n + st[:, None] * (c[:, None] * a + s[:, None] * b))
        q, w = self.turn(c, s, St[:, 1], St[:, 2])
        r12, r33 = -p.p_l * (1.0 - ct * ct) / (1.0 + ct * ct), 2.0 * ct / (1.0 + ct * ct)
        I = St[:, 0].clone()
        St[:, 0], St[:, 1], St[:, 2] = I + r12 * q, r12 * I + q, r33 * w
        a[:] = _unit(torch.linalg.cross(m, n))


def _exact_train(case: dict, seed: int):
    """One training step: loss, gradient (autograd of the stated density), Adam."""
    x, w = (t.double() for t in _training_data(case, seed))
    vec = _warp_params(seed).to("cuda").double().requires_grad_(True)
    z = vec[:32].expand(case["rows"], 32)
    loss, o = 0.0, 32
    centres = (torch.arange(32, device="cuda", dtype=torch.float64) + 0.5) / 32
    blob = lambda t: torch.exp(-0.5 * ((t[:, None] - centres) * 32) ** 2)
    for layer in range(3):
        if layer:  # logits of the conditional: one-blob features through the four-layer network
            h = torch.cat([blob(x[:, 0])] + ([blob(x[:, 1])] if layer == 2 else []), 1)
            for l in range(4):
                out = 32 if l == 3 else 128
                Wl, bl = vec[o:o + out * 128].reshape(out, 128), vec[o + out * 128:o + out * 128 + out]
                o += out * 128 + out
                h = h @ Wl[:, :h.shape[1]].T + bl
                h = torch.relu(h) if l < 3 else h
            z = h
        q = (1.0 - MIX) * torch.softmax(z, 1) + MIX / 32
        b = (x[:, layer] * 32).long().clamp_max(31)
        loss = loss - (w * torch.log(32.0 * q.gather(1, b[:, None]).squeeze(1))).sum() / w.sum()
    g, = torch.autograd.grad(loss, vec)
    m, v = (t.double() for t in _moments(seed))
    m, v = 0.9 * m + 0.1 * g, 0.999 * v + 0.001 * g * g
    t = ADAM_STEP + 1
    new = vec.detach() - ADAM_LR * (m / (1 - 0.9 ** t)) / (torch.sqrt(v / (1 - 0.999 ** t)) + 1e-8)
    return [loss.detach().reshape(1), g, new, m, v]


def exact(case: dict, seed: int):
    kind = case["kind"]
    if kind == "points":
        pts, out = _Points(case["generator"], case["dims"], seed, "cuda"), []
        i = random.Random(seed).randint(1, 1 << 24) + torch.arange(case["count"], device="cuda")
        for d in range(case["dims"]):
            out.append(pts.bits(i, d) if case["fmt"] == "u32" else pts(i, d))
        out = torch.stack(out, 1)
        if case["fmt"] == "u32":  # the values as the 32-bit words they are returned in
            return torch.where(out >= 1 << 31, out - (1 << 32), out).to(torch.int32)
        return out
    if kind == "train":
        return _exact_train(case, seed)
    if kind == "learned":
        return None  # the proposal's bf16 roundings move every packet: another, equally good, sample
    packets = sum(i.n_packets for i in _instances(case, seed)) if kind == "batch" else case["count"]
    steps = packets * case["n"] * (1 + case.get("orders", 0)) * (1 + 0.3 * case.get("observers", 0))
    if steps > EXACT_MOST:
        return None
    grid = _grid(case, seed)
    prob = _problem(case, seed, grid)
    if kind == "batch":
        outs = []
        for i in _instances(case, seed):
            t = _Tracer(prob.replace(albedo=i.albedo, g=i.g), grid)
            view = t.view(i.theta_obs, prob.phi_obs)
            outs.append(t.trace(i.first_index, i.n_packets, [view], kscale=i.kscale)[0, 0] / i.n_packets)
        return torch.stack(outs)
    t = _Tracer(prob, grid)
    angles = _angles(case, seed) if kind == "observers" else [(prob.theta_obs, prob.phi_obs)]
    img = t.trace(_first(case, seed), case["count"], [t.view(*a) for a in angles]) / case["count"]
    return list(img) if kind == "observers" else img[0]


EXACT_MOST = 4e9  # packet-cells of a 64-bit trace that take about twenty seconds

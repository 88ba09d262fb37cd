"""The work a user has this framework do, as cases that can be timed and compared.

A case is one pass through the public entry points of
``paper_2304_05639_gb300.lenia`` on a seeded synthetic world: a step, a
rollout, an evolution step, a differentiable rollout with its backward pass, a
rollout of many worlds at once, or a step from host buffers.  ``listed()``
names twelve of them, ``draw(rng)`` gives more of the same ranges, ``exact()``
restates each pass in 64 bits with plain torch and numpy.
"""
import math

import numpy as np
import torch

from paper_2304_05639_gb300 import inputs, lenia

HALF_HEIGHT = 1.1774100225154747   # sqrt(2 ln 2): where exp(-z^2 / 2) = 1/2


def _case(name=None, **kw):
    c = dict(kind="step", H=1024, W=1024, C=1, n_self=3, R=12, loc=3, maintain=1, r_diff=1, alpha_on=0,
             rings=0, steps=1, dt=0.1, patch=128, geno=16, worlds=0)
    c.update(kw)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # the smallest world of the benchmark: one kernel, global genes, a short
        # rollout (an interactive view of a filled torus); launches and latency count
        _case("small_rollout_64", kind="rollout", H=64, W=64, n_self=1, R=13, loc=0, maintain=0, steps=16, patch=64,
              geno=1),
        # the benchmark's one-channel world with per-site genes, stepped on
        _case("rollout_1024", kind="rollout", n_self=1, steps=6),
        # the headline: the paper's 3-channel, 15-kernel topology with gene maps,
        # one step with its statistics
        _case("paper_step_2048", H=2048, W=2048, C=3, R=18, dt=0.2, patch=256),
        # the same topology on a screen-shaped torus (no side a power of two)
        _case("screen_step_1080x1920", H=1080, W=1920, C=3, R=13, dt=0.2, patch=192),
        # a small ragged one-channel world, stepped on
        _case("ragged_rollout_300x404", kind="rollout", H=300, W=404, n_self=1, steps=6, patch=64, geno=8),
        # short-range kernels (the benchmark's R = 5 world)
        _case("short_range_step_2048", H=2048, W=2048, C=3, R=5, dt=0.2, patch=256),
        # ring-wise kernel genes: the paper's 512 x 1024 configuration, every
        # gene type per site (135 gene planes)
        _case("rings_step_512x1024", H=512, W=1024, C=3, R=12, loc=15, rings=24, alpha_on=1, dt=0.2, patch=96, geno=8),
        # two channels (8 kernels) with mu, sigma and h per site and a wider
        # diffusion disk: a world outside the paper's own layout
        _case("two_channel_step_512", H=512, W=512, C=2, R=12, loc=7, r_diff=2, patch=96, geno=8),
        # an evolution step: walls, mutation and penalisation around the step
        _case("evolve_step_1024", kind="evolve", H=1024, W=1024, C=3, R=18, dt=0.2),
        # the differentiable rollout and its backward pass (gene and
        # initial-state gradients), checkpoints every 8 steps
        _case("adjoint_256", kind="adjoint", H=256, W=256, C=3, R=13, loc=0, maintain=0, steps=12, dt=0.02,
              patch=96, geno=1),
        # many independent worlds of uneven sizes advanced together
        _case("batch_64_worlds", kind="batch", H=512, W=512, n_self=1, steps=4, worlds=64, geno=4),
        # a serving call: a step from page-locked host buffers and back
        _case("host_step_512", kind="host", H=512, W=512, C=3, R=18, dt=0.2, patch=96, geno=8),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _sides(rng, lo, hi):
    """A torus: half of them square powers of two, half of any shape (W a multiple of 4)."""
    if rng.random() < 0.5:
        p = [n for n in (64, 128, 256, 512, 1024, 2048) if lo <= n <= hi]
        return rng.choice(p), rng.choice(p)
    return _log_int(rng, lo, hi), max(lo, _log_int(rng, lo, hi) // 4 * 4)


def _patch(H, W):
    return max(16, int(math.sqrt(H * W)) // 6)


def draw(rng):
    kind = rng.choice(["step", "step", "step", "rollout", "rollout", "rings", "evolve", "adjoint", "batch", "host"])
    R = rng.randint(4, 20)
    common = dict(R=R, geno=rng.randint(2, 16), alpha_on=int(rng.random() < 0.25))
    if kind == "rollout":
        if rng.random() < 0.4:
            H, W = rng.choice([(64, 64), (64, 128), (128, 128), (96, 80), (128, 256)])
            return _case(kind="rollout", H=H, W=W, n_self=1, loc=0, maintain=0, steps=rng.randint(2, 16),
                         patch=min(H, W),
                         **{**common, "geno": 1, "alpha_on": 0})
        H, W = _sides(rng, 64, 2048)
        return _case(kind="rollout", H=H, W=W, n_self=1, steps=rng.randint(2, 6), patch=_patch(H, W),
                     **common)
    if kind == "rings":
        H, W = _sides(rng, 64, 768)
        return _case(H=H, W=W, C=3, loc=15, rings=rng.choice([12, 24]), dt=0.2, patch=_patch(H, W),
                     **{**common, "alpha_on": 1, "R": rng.choice([6, 12])})
    if kind == "adjoint":
        H, W = _sides(rng, 64, 512)
        return _case(kind="adjoint", H=H, W=W, C=rng.choice([1, 3]), loc=0, maintain=0, steps=rng.randint(2, 12),
                     dt=0.02, patch=2 * _patch(H, W), **{**common, "geno": 1, "alpha_on": 0})
    if kind == "batch":
        return _case(kind="batch", H=512, W=512, n_self=1, steps=rng.randint(2, 4), worlds=_log_int(rng, 8, 64),
                     **{**common, "geno": 4})
    if kind == "host":
        H, W = _sides(rng, 64, 768)
        return _case(kind="host", H=H, W=W, C=rng.choice([1, 3]), dt=0.2, patch=_patch(H, W), **common)
    # steps and evolution steps: 1 to 4 channels, at most the headline's gene planes
    C = rng.choice([1, 2, 3, 3, 3, 4])
    n_self = rng.choice([1, 2, 3, 3])
    loc = rng.choice([3, 3, 3, 7, 0]) if kind == "step" else rng.choice([3, 3, 7])
    H, W = _sides(rng, 64, 2048)
    K = C * n_self + C * (C - 1)
    while H * W * K * max(1, bin(loc).count("1")) > 2048 * 2048 * 30:
        H, W = max(64, H // 2), max(64, W // 2 // 4 * 4)
    return _case(kind=kind, H=H, W=W, C=C, n_self=n_self, loc=loc, maintain=int(loc != 0),
                 r_diff=rng.choice([1, 1, 1, 2]), dt=0.2, patch=_patch(H, W), **common)


# ---------------------------------------------------------------- inputs

def _kernels(case, nrng):
    """The world's kernels: random shells (or, with rings, two bumps whose genes
    the maps replace) in the paper's topology."""
    ks = []
    for s, d in inputs.paper_topology(case["C"], case["n_self"]):
        if case["rings"]:
            ks.append(inputs.KernelDesc(s, d, case["R"], inputs.KERNEL_BUMPS, (1.0,), bump=(0.3, 0.1, 0.8, 0.7, 0.1, 0.3),
                                        h=0.6))
            continue
        B = int(nrng.integers(1, 4)) if case["C"] > 1 else 1
        beta = tuple(float(b) for b in nrng.uniform(0.25, 1.0, B))
        h = float(np.float32(nrng.uniform(0.1, 1.0))) if case["C"] > 1 else 1.0
        ks.append(inputs.KernelDesc(s, d, case["R"], inputs.KERNEL_SHELLS, beta, h=h))
    return ks


def _genotypes(case, ks, nrng):
    """Levels [G][C] and gene values {plane: [G][K]}: every kernel's bump sits
    beside the potential its patch starts with, so that the patches live."""
    G, K = case["geno"], len(ks)
    level = nrng.uniform(0.10, 0.40, (G, case["C"]))
    src = np.array([k.src for k in ks])
    sigma = nrng.uniform(0.03, 0.06, (G, K))
    g = {"mu": level[:, src] + nrng.uniform(-0.01, 0.01, (G, K)) - HALF_HEIGHT * sigma, "sigma": sigma,
         "h": np.tile([k.h for k in ks], (G, 1))}
    for n, (lo, hi) in {"r1": (0.1, 0.5), "w1": (0.05, 0.15), "b1": (0.5, 1.0), "r2": (0.5, 0.9), "w2": (0.05, 0.15),
                        "b2": (0.1, 0.6)}.items():
        g[n] = nrng.uniform(lo, hi, (G, K))
    return level, g


def _world(case, seed, device):
    """(inputs.World without state, A [C][H][W], P [n_p][K][H][W] or None)."""
    nrng = np.random.default_rng(seed)
    H, W, C, R = case["H"], case["W"], case["C"], case["R"]
    ks = _kernels(case, nrng)
    level, genes = _genotypes(case, ks, nrng)
    for k, kd in enumerate(ks):
        kd.mu, kd.sigma = float(np.float32(genes["mu"][0, k])), float(np.float32(genes["sigma"][0, k]))
    w = inputs.World(H, W, C, ks, case["dt"], localized=case["loc"], maintain_genes=case["maintain"],
                     r_diff=case["r_diff"], alpha_on=case["alpha_on"], n_rings=case["rings"])
    # the genotype of each site: patches at random places, later ones on top
    body = torch.full((H, W), -1, dtype=torch.long)
    maps = torch.full((H, W), -1, dtype=torch.long)
    for g in range(case["geno"]):
        cy, cx = int(nrng.integers(0, H)), int(nrng.integers(0, W))
        if case["geno"] == 1:
            cy, cx = H // 2, W // 2
        half = case["patch"] // 2
        for m, n in ((body, half), (maps, half + R)):
            ys = torch.arange(cy - n, cy + n) % H
            xs = torch.arange(cx - n, cx + n) % W
            m[ys[:, None], xs[None, :]] = g
    body, maps = body.to(device), maps.to(device)
    gen = torch.Generator(device="cpu").manual_seed(seed)
    A = torch.rand((C, H, W), generator=gen, dtype=torch.float32).to(device)
    scale = torch.cat([torch.from_numpy(2.0 * level), torch.zeros(1, C, dtype=torch.float64)]).float().to(device)
    A *= scale.t()[:, body]
    names = [n for n, b in (("mu", 1), ("sigma", 2), ("h", 4)) if case["loc"] & b]
    if case["loc"] & 8:
        names += ["r1", "w1", "b1", "r2", "w2", "b2"]
    P = None
    if names:
        P = torch.empty((len(names), len(ks), H, W), dtype=torch.float32, device=device)
        for i, n in enumerate(names):
            v = np.concatenate([genes[n], np.zeros((1, len(ks)))]).astype(np.float32)
            P[i] = torch.from_numpy(v).to(device).t()[:, maps]
    return w, A, P


def _events(case, seed):
    """One step's mutation and penalisation, and a vertical wall."""
    nrng = np.random.default_rng(seed + 77)
    K = len(inputs.paper_topology(case["C"], case["n_self"]))
    H, W = case["H"], case["W"]
    ev = dict(mut_p=0, mut_k=int(nrng.integers(0, K)), mut_x0=int(nrng.integers(0, W)), mut_y0=int(nrng.integers(0, H)),
              mut_half=16, mut_delta=float(nrng.uniform(-0.01, 0.01)), gamma_mut=1.0, pen_p=1,
              pen_k=int(nrng.integers(0, K)), pen_delta=-float(nrng.uniform(0.002, 0.01)), gamma_pen=0.2, eps_pen=0.5,
              r_oxy=4)
    mask = np.zeros((H, W), np.uint8)
    x0 = int(nrng.integers(0, W - 8))
    mask[:, x0:x0 + 8] = 1
    return ev, mask


def _batch_cases(case):
    """One-channel worlds with sides of 64 to 512 and radii of 8 to 16."""
    return [_case(H=S, W=S, n_self=1, R=8 + 5 * i % 9, alpha_on=case["alpha_on"], geno=case["geno"], patch=max(8, S // 4))
            for i, S in enumerate([64, 128, 256, 512][j % 4] for j in range(case["worlds"]))]


class _State:
    """What a user's program holds: the handle and the world's buffers."""

    def __init__(self, kind):
        self.kind, self.ctx, self.batch, self.fn = kind, None, None, None

    def __del__(self):
        lenia.lenia_destroy(self.ctx)
        lenia.lenia_batch_destroy(self.batch)


def prepare(case, seed):
    kind = case["kind"]
    st = _State(kind)
    st.steps = case["steps"]
    if kind == "batch":
        made = [_world(c, seed * 1009 + i, "cpu") for i, c in enumerate(_batch_cases(case))]
        worlds = [w for w, _, _ in made]
        # every world's state in one buffer, world after world
        st.A0 = torch.cat([A.reshape(-1) for _, A, _ in made]).cuda()
        st.P0 = torch.cat([P.reshape(-1) for _, _, P in made]).cuda()
        st.A, st.P = torch.empty_like(st.A0), torch.empty_like(st.P0)
        st.views = [list(b.split([m[i].numel() for m in made])) for i, b in ((1, st.A), (2, st.P))]
        st.batch = lenia.lenia_batch_init(worlds)
        return st
    w, A, P = _world(case, seed, "cuda")
    if kind == "adjoint":
        st.fn = lenia.LeniaRollout(w, case["steps"], ckpt_every=8)
        st.A0 = A
        st.genes = torch.from_numpy(lenia.genes_of(w)).cuda()
        gen = torch.Generator(device="cpu").manual_seed(seed + 1)
        st.gA = torch.randn(A.shape, generator=gen).cuda()
        return st
    cfg, ks = lenia.config_from_world(w)
    st.ctx = lenia.lenia_init(cfg, ks)
    st.A0, st.P0 = A, P
    st.A = torch.empty_like(A)
    st.P = torch.empty_like(P) if P is not None else None
    st.stats = torch.zeros((case["C"], 3), dtype=torch.float32, device="cuda")
    if kind == "evolve":
        ev, mask = _events(case, seed)
        st.ev = lenia.events_struct(ev)
        lenia.lenia_set_walls(st.ctx, mask)
    if kind == "host":
        st.A0 = A.cpu().pin_memory()
        st.P0 = P.cpu().pin_memory()
        st.A = torch.empty_like(st.A0, pin_memory=True)
        st.P = torch.empty_like(st.P0, pin_memory=True)
        st.stats = torch.zeros((case["C"], 3), dtype=torch.float32, pin_memory=True)
    return st


def run(st):
    if st.kind == "step":
        lenia.lenia_step(st.ctx, st.A0, st.P0, st.A, st.P, st.stats)
        return [st.A, st.P, st.stats]
    if st.kind == "rollout":
        # the rollout advances its buffers in place: it starts from a copy
        st.A.copy_(st.A0)
        if st.P is not None:
            st.P.copy_(st.P0)
        lenia.lenia_rollout(st.ctx, st.A, st.P, st.steps)
        return [st.A, st.P]
    if st.kind == "evolve":
        lenia.lenia_step_evolve(st.ctx, st.A0, st.P0, st.A, st.P, st.ev, st.stats)
        return [st.A, st.P, st.stats]
    if st.kind == "adjoint":
        A0 = st.A0.requires_grad_(True)
        genes = st.genes.requires_grad_(True)
        A0.grad = genes.grad = None
        A = st.fn(A0, genes)
        A.backward(st.gA)
        return [A.detach(), A0.grad, genes.grad]
    if st.kind == "batch":
        st.A.copy_(st.A0)
        st.P.copy_(st.P0)
        lenia.lenia_batch_rollout(st.batch, *st.views, st.steps)
        return [st.A, st.P]
    lenia.lenia_step_host(st.ctx, st.A0, st.P0, st.A, st.P, st.stats)
    return [st.A, st.P, st.stats]


def _planes(case):
    """(convolved channels, convolution outputs, gene planes) of a world."""
    K = len(inputs.paper_topology(case["C"], case["n_self"]))
    n_p = bin(case["loc"] & 7).count("1") + (6 if case["loc"] & 8 else 0)
    return case["C"], (case["C"] * case["rings"] if case["rings"] else K), n_p * K


def work(case):
    """The state in and out once; the real transforms of every step's
    convolutions counted the standard way (5 n log2 n, half for real data)."""
    if case["kind"] == "batch":
        n = float(sum(c["H"] * c["W"] for c in _batch_cases(case)))
        return {"bytes": n * 24.0, "flops": n * case["steps"] * 2 * 2.5 * 17.5}
    C, K, G = _planes(case)
    n = case["H"] * case["W"]
    conv = 2.5 * math.log2(n)
    passes = case["steps"]
    if case["kind"] == "adjoint":
        # forward; then, per reversed step, the K gradient planes in and C out
        return {"bytes": n * C * 16.0, "flops": n * passes * conv * 2 * (C + K)}
    return {"bytes": n * (C + G) * 8.0, "flops": n * passes * conv * (C + K)}


# ------------------------------------------------- the same passes in 64 bits

def _offsets(R, device):
    d = torch.arange(-R, R + 1, dtype=torch.float64, device=device)
    return d[:, None].square() + d[None, :].square()


def _weights(kd, device):
    """The normalised kernel [2R+1][2R+1] (Section 2.1 and the original shells)."""
    rho = _offsets(kd.radius, device).sqrt() / kd.radius
    if kd.form == inputs.KERNEL_SHELLS:
        br = rho * len(kd.beta)
        i = br.floor().clamp(max=len(kd.beta) - 1).long()
        q = br - br.floor()
        inner = (q > 0) & (q < 1)
        qs = torch.where(inner, q, torch.full_like(q, 0.5))
        k = torch.where(inner, torch.exp(4 - 1 / (qs * (1 - qs))), torch.zeros_like(q))
        k = k * torch.tensor(kd.beta, dtype=torch.float64, device=device)[i]
    else:
        k = sum(kd.bump[3 * b + 2] * torch.exp(-(rho - kd.bump[3 * b]).square() / (2 * kd.bump[3 * b + 1] ** 2))
                for b in (0, 1))
    k = torch.where(rho < 1, k, torch.zeros_like(k))
    return k / k.sum()


def _spectrum(k, H, W):
    """rfft2 of a centred kernel laid on the torus."""
    R = k.shape[0] // 2
    f = torch.zeros((H, W), dtype=torch.float64, device=k.device)
    idx = torch.arange(-R, R + 1, device=k.device)
    f.index_put_(((idx % H)[:, None].expand_as(k), (idx % W)[None, :].expand_as(k)), k, accumulate=True)
    return torch.fft.rfft2(f)


def _spectra(w, device):
    if not w.n_rings:
        return [_spectrum(_weights(kd, device), w.height, w.width) for kd in w.kernels], None
    R, n = w.kernels[0].radius, w.n_rings
    d2 = _offsets(R, device)
    # ring r: r <= n |d| / R < r + 1, |d| < R, decided on integers (n^2 d^2 against m^2 R^2)
    edges = torch.arange(1, n + 1, dtype=torch.float64, device=device).square() * R * R
    ring = torch.bucketize(n * n * d2, edges, right=True)
    masks = [((ring == r) & (d2 < R * R)).double() for r in range(n)]
    return [_spectrum(m, w.height, w.width) for m in masks], torch.stack([m.sum() for m in masks])


def _disk_sum(x, r):
    out = torch.zeros_like(x)
    for dy in range(-r, r + 1):
        for dx in range(-r, r + 1):
            if dy * dy + dx * dx <= r * r:
                out += torch.roll(x, (dy, dx), (-2, -1))
    return out


def _step64(w, spec, cnt, A, P, events=None):
    """One step (Algorithm 2: diffuse .. update), with the evolutionary lines
    where events = (ev, wall mask) are given.  Plane by plane, to bound memory."""
    H, W, K = w.height, w.width, w.n_kernels
    if events:
        keep = torch.from_numpy(events[1] == 0).to(A.device)
        A, P = A * keep, P * keep
    FA = torch.fft.rfft2(A)
    Pd = P
    if P is not None and w.maintain_genes:
        Pd = torch.empty_like(P)
        for p in range(P.shape[0]):
            s = _disk_sum(P[p], w.r_diff)
            n = _disk_sum((P[p] > w.eps_p).double(), w.r_diff)
            Pd[p] = torch.where(n > 0, (s / n.clamp(min=1)).clamp(0, 1), torch.zeros_like(s))
    alpha = torch.ones((H, W), dtype=torch.bool, device=A.device)
    n_growth = bin(w.localized & 7).count("1")
    order = [i for i, b in ((0, 1), (1, 2), (2, 4)) if w.localized & b]

    def gene(i, k, value):
        return Pd[order.index(i), k] if i in order else torch.full((), float(np.float32(value)), device=A.device,
                                                                   dtype=torch.float64)

    acc = torch.zeros_like(A)
    off = [0.0] * w.n_channels
    tsum = torch.zeros((H, W), dtype=torch.float64, device=A.device)
    V, vsrc = None, -1
    for k in sorted(range(K), key=lambda k: w.kernels[k].src):
        kd = w.kernels[k]
        if w.n_rings:
            if vsrc != kd.src:
                V, vsrc = torch.fft.irfft2(FA[kd.src] * torch.stack(spec), s=(H, W)), kd.src
            r1, w1, b1, r2, w2, b2 = (Pd[n_growth + i, k] for i in range(6))
            num = torch.zeros_like(tsum)
            den = torch.zeros_like(tsum)
            for r in range(w.n_rings):
                x = r / w.n_rings
                kr = sum(torch.where(ww > 0, b * torch.exp(-(x - c).square() / (2 * torch.where(ww > 0, ww, torch.ones_like(ww)).square())),
                                     torch.zeros_like(b)) for c, ww, b in ((r1, w1, b1), (r2, w2, b2)))
                num += kr * V[r]
                den += kr * cnt[r]
            U = torch.where(den > 0, num / torch.where(den > 0, den, torch.ones_like(den)), torch.zeros_like(num))
        else:
            U = torch.fft.irfft2(FA[kd.src] * spec[k], s=(H, W))
        m, sg, h = gene(0, k, kd.mu), gene(1, k, kd.sigma), gene(2, k, kd.h)
        g = torch.where(sg > 0, torch.exp(-((U - m) / torch.where(sg > 0, sg, torch.ones_like(sg))).square() / 2),
                        torch.zeros_like(U))
        t = U if w.alpha_on else h * g
        tsum += t
        if w.maintain_genes:
            alpha &= t > float(np.float32(w.eps_u))
        acc[kd.dst] = acc[kd.dst] + h * (2 * g - 1)
        if 2 not in order:
            off[kd.dst] -= float(np.float32(kd.h))
    dt = float(np.float32(w.dt))
    if w.maintain_genes:
        for p in range(Pd.shape[0]):
            alpha &= (Pd[p] > w.eps_p).all(dim=0)
        base = torch.tensor(off, dtype=torch.float64, device=A.device)[:, None, None].expand_as(acc)
        acc = torch.where(alpha, acc, base)
        Pd = Pd * alpha
    A1 = (A + dt * acc).clamp(0, 1)
    if events:
        ev = events[0]
        r = ev["r_oxy"]
        empty = (tsum <= float(np.float32(w.eps_u))).double()
        n = float((_offsets(r, "cpu") <= r * r).sum())
        M = _disk_sum(n - _disk_sum(empty, r), r)
        y = torch.arange(H, device=A.device)
        x = torch.arange(W, device=A.device)
        half = ev["mut_half"]
        sq = ((y - ev["mut_y0"] + half) % H < 2 * half)[:, None] & ((x - ev["mut_x0"] + half) % W < 2 * half)[None, :]
        Pd[ev["mut_p"], ev["mut_k"]] += ev["gamma_mut"] * ev["mut_delta"] * (sq & alpha)
        Pd[ev["pen_p"], ev["pen_k"]] += ev["gamma_pen"] * ev["pen_delta"] * ((M > ev["eps_pen"] * n * n) & alpha)
    return A1, Pd


def _stats64(A):
    out = []
    for a in A:
        row = [a.sum()]
        for dim, n in ((0, A.shape[1]), (1, A.shape[2])):
            m = a.sum(dim=1 - dim)
            t = 2 * math.pi * torch.arange(n, dtype=torch.float64, device=A.device) / n
            c = torch.atan2((m * t.sin()).sum(), (m * t.cos()).sum()) * n / (2 * math.pi)
            row.append(torch.where(c < 0, c + n, c))
        out.append(torch.stack(row))
    return torch.stack(out)


def _rollout64(case, seed, device, steps, events=None):
    w, A, P = _world(case, seed, device)
    spec, cnt = _spectra(w, device)
    A, P = A.double(), (P.double() if P is not None else None)
    for _ in range(steps):
        A, P = _step64(w, spec, cnt, A, P, events)
    return A, P


def exact(case, seed):
    device = "cuda" if torch.cuda.is_available() else "cpu"
    kind = case["kind"]
    if kind == "batch":
        out = [_rollout64(c, seed * 1009 + i, device, case["steps"]) for i, c in enumerate(_batch_cases(case))]
        return [torch.cat([o[j].reshape(-1) for o in out]) for j in (0, 1)]
    if kind == "adjoint":
        w, A0, _ = _world(case, seed, device)
        spec, _ = _spectra(w, device)
        genes = torch.from_numpy(lenia.genes_of(w)).double().to(device).requires_grad_(True)
        gen = torch.Generator(device="cpu").manual_seed(seed + 1)
        gA = torch.randn(A0.shape, generator=gen).double().to(device)
        a0 = A0.double().requires_grad_(True)
        src = [kd.src for kd in w.kernels]
        dst = torch.tensor([kd.dst for kd in w.kernels], device=device)
        S = torch.stack(spec)
        A = a0
        for _ in range(case["steps"]):
            U = torch.fft.irfft2(torch.fft.rfft2(A)[src] * S, s=(w.height, w.width))
            mu, sg, h = (genes[:, i, None, None] for i in range(3))
            G = h * (2 * torch.exp(-((U - mu) / sg).square() / 2) - 1)
            A = (A + float(np.float32(w.dt)) * torch.zeros_like(A).index_add(0, dst, G)).clamp(0, 1)
        A.backward(gA)
        return [A.detach(), a0.grad, genes.grad]
    ev = _events(case, seed) if kind == "evolve" else None
    A, P = _rollout64(case, seed, device, case["steps"] if kind == "rollout" else 1, ev)
    return [A, P] if kind == "rollout" else [A, P, _stats64(A)]

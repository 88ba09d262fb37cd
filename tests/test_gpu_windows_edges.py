"""The windows and the per-site update kernel off the usual worlds: channels that
no kernel reads, narrow bumps and large radii (every alpha decision is that of
the direct sums), values outside [0, 1], infinite genes, long sums, and groups
of worlds.  GPU only."""
import dataclasses

import numpy as np
import pytest

import oracle
from paper_2304_05639_gb300 import build, inputs, lenia
from gpu_util import TOL_U, gpu_potentials, to_dev, torch_mod

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    build.build()
    oracle.build()
    torch_mod()


def _gradients(w, n_steps, path):
    torch = torch_mod()
    f = lenia.LeniaRollout(w, n_steps, ckpt_every=2, conv_path=path)
    A = to_dev(w.A).requires_grad_(True)
    genes = torch.from_numpy(lenia.genes_of(w)).cuda().requires_grad_(True)
    gen = torch.Generator().manual_seed(3)
    f(A, genes).backward(torch.randn(w.A.shape, generator=gen).cuda())
    f.close()
    return A.grad.double(), genes.grad.double()


def _gradients64(w, n_steps):
    """The same in 64 bits: plain torch, convolutions in the frequency domain."""
    torch = torch_mod()
    spec = []
    for k, kw in zip(w.kernels, oracle.world_kernels(w)):
        f = torch.zeros((w.height, w.width), dtype=torch.float64)
        i = torch.arange(-k.radius, k.radius + 1)
        f.index_put_(((i % w.height)[:, None], (i % w.width)[None, :]), torch.from_numpy(kw), accumulate=True)
        spec.append(torch.fft.rfft2(f).cuda())
    A0 = to_dev(w.A).double().requires_grad_(True)
    genes = torch.from_numpy(lenia.genes_of(w)).cuda().double().requires_grad_(True)
    A = A0
    for _ in range(n_steps):
        acc = [torch.zeros_like(A[0]) for _ in range(w.n_channels)]
        for k, (kd, S) in enumerate(zip(w.kernels, spec)):
            U = torch.fft.irfft2(torch.fft.rfft2(A[kd.src]) * S, s=(w.height, w.width))
            mu, sigma, h = genes[k]
            acc[kd.dst] = acc[kd.dst] + h * (2 * torch.exp(-0.5 * ((U - mu) / sigma) ** 2) - 1)
        A = (A + w.dt * torch.stack(acc)).clamp(0, 1)
    gen = torch.Generator().manual_seed(3)
    A.backward(torch.randn(w.A.shape, generator=gen).cuda().double())
    return A0.grad, genes.grad


@pytest.mark.parametrize("shape,topology", [((100, 72, 9), [(0, 1)]), ((64, 64, 9), [(0, 1)]), ((130, 140, 13), [(0, 0), (0, 1)]),
                                            ((300, 404, 12), [(1, 0), (1, 2), (1, 1)]), ((128, 128, 20), [(2, 0)])])
def test_gradient_of_channels_that_no_kernel_reads(shape, topology):
    """dL/dA_0 of a channel that is only written is the carried gradient itself
    (relative 2-norm 1e-4 per channel and of the genes' gradients, against 64 bits)."""
    H, W, R = shape
    C = max(max(t) for t in topology) + 1
    ks = [inputs.KernelDesc(s, d, R, inputs.KERNEL_SHELLS, (1.0,), h=0.7, mu=0.5, sigma=0.08) for s, d in topology]
    # (three updates of at most 0.02 x 0.7 x 3: no site comes near a clip, whose two
    # sides differ by a whole gradient)
    w = inputs.World(H, W, C, ks, 0.02, localized=0, maintain_genes=0)
    w.A = (0.3 + 0.4 * inputs.random_field(H + W, (C, H, W))).astype(np.float32)
    (a, ga), (b, gb) = _gradients(w, 3, lenia.CONV_AUTO), _gradients64(w, 3)
    for c in range(C):
        print("channel", c, float((a[c] - b[c]).norm() / b[c].norm()))
        assert float((a[c] - b[c]).norm()) <= 1e-4 * float(b[c].norm())
    print("genes", float((ga - gb).norm() / gb.norm()))
    assert float((ga - gb).norm()) <= 1e-4 * float(gb.norm())


def _potentials_of(w, path, A):
    g = inputs.World(w.height, w.width, w.n_channels, w.kernels, w.dt, localized=0, maintain_genes=0)
    return gpu_potentials(g, path, A)[0]


def _decisions(w, path):
    """(alpha, E_pen) of one evolution step without mutation or penalisation."""
    torch = torch_mod()
    ev = inputs.evolution_events(w, 0, gamma_mut=0.0, gamma_pen=0.0)
    cfg, ks = lenia.config_from_world(w, path)
    ctx = lenia.lenia_init(cfg, ks)
    try:
        A, P = to_dev(w.A), to_dev(w.P) if w.n_planes else None
        A2, P2 = torch.empty_like(A), torch.empty_like(P) if w.n_planes else None
        al = torch.zeros((w.height, w.width), dtype=torch.uint8, device="cuda")
        ep = torch.zeros((w.height, w.width), dtype=torch.float32, device="cuda")
        lenia.lenia_step_evolve(ctx, A, P, A2, P2, ev, None, al, ep)
        torch.cuda.synchronize()
        return al.cpu().numpy(), ep.cpu().numpy()
    finally:
        lenia.lenia_destroy(ctx)


def _uniform_at_threshold(w, sigma, z, on_windows, n_levels=24):
    """Makes a uniform world of w, at the level (of n_levels) where the direct sums'
    one potential and the windows' are furthest apart.  Returns (mu, eps_u): a bump
    of width sigma z widths above the windows' (or the sums') potential, and a
    threshold half-way between the two routes' bumps."""
    best = None
    for level in np.linspace(0.3, 1.0, n_levels):
        A = np.full(w.A.shape, level, np.float32)
        d, t = (_potentials_of(w, p, A) for p in (lenia.CONV_DIRECT, lenia.CONV_AUTO))
        assert (d == d.flat[0]).all()
        ud, uw = float(d.flat[0]), float(t.mean(dtype=np.float64))
        if best is None or abs(ud - uw) > abs(best[0] - best[1]):
            best = ud, uw, A
    ud, uw, w.A = best
    assert ud != uw
    mu = np.float32((uw if on_windows else ud) - z * sigma)
    bump = lambda v: np.exp(-0.5 * ((v - float(mu)) / float(np.float32(sigma))) ** 2)
    print("direct", ud, "windows", uw, "bumps", bump(ud), bump(uw))
    return mu, 0.5 * (bump(ud) + bump(uw))


@pytest.mark.parametrize("sigma", [2e-4, 3e-4, 6e-4, 2e-3])
@pytest.mark.parametrize("z", [0.0, 0.01, 0.2, 2.0])
@pytest.mark.parametrize("on_windows", [False, True])
def test_narrow_bumps_decide_as_the_direct_sums(sigma, z, on_windows):
    w = inputs.localized_single_channel(H=130, W=132, R=31, patch=64, n_geno=1, live=True)
    w.P[0], w.eps_u = _uniform_at_threshold(w, sigma, z, on_windows)
    w.P[1] = np.float32(sigma)
    a, b = _decisions(w, lenia.CONV_AUTO), _decisions(w, lenia.CONV_DIRECT)
    np.testing.assert_array_equal(a[0], b[0])
    np.testing.assert_array_equal(a[1], b[1])


FLAT = inputs.KernelDesc(0, 0, 1, inputs.KERNEL_BUMPS, (1.0,), bump=(0.0, 1e5, 1.0, 0.5, 0.1, 0.0))
SHELL = inputs.KernelDesc(0, 0, 1, inputs.KERNEL_SHELLS, (1.0,))
SIGNED = inputs.KernelDesc(0, 0, 1, inputs.KERNEL_SHELLS, (-0.4, 1.0))      # absolute weights sum to more than 1


# (300 x 512: the streaming kernel's arithmetic)
@pytest.mark.parametrize("shape", [(130, 132, 12), (300, 404, 20), (300, 512, 20), (300, 404, 31), (600, 900, 56)])
@pytest.mark.parametrize("kernel", [FLAT, SHELL, SIGNED], ids=["flat", "shell", "signed"])
@pytest.mark.parametrize("sigma,z", [(0.03, 1.0), (0.004, 0.0)])
@pytest.mark.parametrize("on_windows", [False, True])
def test_the_sums_rounding_at_any_radius(shape, kernel, sigma, z, on_windows):
    """The direct sums' rounding grows with their taps, most with equal weights (a flat
    disk: 1.5e-5 at R = 20, 1.4e-4 at R = 56): the decisions are still theirs."""
    H, W, R = shape
    w = inputs.localized_single_channel(H=H, W=W, R=R, patch=64, n_geno=1, live=True)
    w.kernels = [dataclasses.replace(w.kernels[0], form=kernel.form, beta=kernel.beta, bump=kernel.bump)]
    w.P[0], w.eps_u = _uniform_at_threshold(w, sigma, z, on_windows)
    w.P[1] = np.float32(sigma)
    a, b = _decisions(w, lenia.CONV_AUTO), _decisions(w, lenia.CONV_DIRECT)
    np.testing.assert_array_equal(a[0], b[0])
    np.testing.assert_array_equal(a[1], b[1])


@pytest.mark.parametrize("eps_u", [0.0, 0.01])
def test_evolution_on_a_mostly_empty_world_costs_no_more_than_direct_sums(eps_u):
    """Sites without genes need no settling: their tests are zero on both routes."""
    torch = torch_mod()
    w = inputs.multi_channel(H=540, W=960, R=13, patch=64, n_geno=3, matched=True)
    w.eps_u = eps_u
    a, b = _decisions(w, lenia.CONV_AUTO), _decisions(w, lenia.CONV_DIRECT)
    np.testing.assert_array_equal(a[0], b[0])
    np.testing.assert_array_equal(a[1], b[1])
    ev = inputs.evolution_events(w, 0)
    us = []
    for path in (lenia.CONV_AUTO, lenia.CONV_DIRECT):
        cfg, ks = lenia.config_from_world(w, path)
        ctx = lenia.lenia_init(cfg, ks)
        A, P = to_dev(w.A), to_dev(w.P)
        A2, P2 = torch.empty_like(A), torch.empty_like(P)
        t = []
        for i in range(8):
            e0, e1 = (torch.cuda.Event(enable_timing=True) for _ in range(2))
            e0.record()
            lenia.lenia_step_evolve(ctx, A, P, A2, P2, ev)
            e1.record()
            torch.cuda.synchronize()
            t.append(e0.elapsed_time(e1) * 1e3)
        lenia.lenia_destroy(ctx)
        us.append(float(np.median(t[3:])))
    print("evolution step us, windows and direct sums:", us)
    assert us[0] <= us[1]


@pytest.mark.parametrize("z", [14.0, 14.35, 14.4, 15.5])
def test_thresholds_at_zero_decide_as_the_direct_sums(z):
    """eps_u = 0: the decision lies where a bump underflows."""
    w = inputs.localized_single_channel(H=130, W=132, R=31, patch=64, n_geno=1, live=True)
    rng = np.random.default_rng(3)
    w.A = (0.5 + 0.02 * rng.standard_normal(w.A.shape)).clip(0, 1).astype(np.float32)
    w.P[0], w.P[1], w.eps_u = np.float32(0.5 - z * 0.03), np.float32(0.03), 0.0
    a, b = _decisions(w, lenia.CONV_AUTO), _decisions(w, lenia.CONV_DIRECT)
    print("alpha", b[0].mean())
    np.testing.assert_array_equal(a[0], b[0])
    np.testing.assert_array_equal(a[1], b[1])


def _near(H, W, y, x, R):
    """Sites of a torus within |d| < R of (y, x)."""
    dy = np.minimum((np.arange(H) - y) % H, (y - np.arange(H)) % H)
    dx = np.minimum((np.arange(W) - x) % W, (x - np.arange(W)) % W)
    return dy[:, None] ** 2 + dx[None, :] ** 2 < R * R


@pytest.mark.parametrize("localized", [3, 7])
@pytest.mark.parametrize("r_diff", [1, 2])
@pytest.mark.parametrize("value", [np.inf, 3e38, 40.0])
def test_diffused_genes_saturate(localized, r_diff, value):
    """A gene above the disk's count diffuses to 1, an infinite one too."""
    torch = torch_mod()
    w = inputs.multi_channel(H=72, W=100, R=9, patch=40, n_geno=4, matched=True, localized=localized, seed_index=31,
                             n_channels=2)
    w.r_diff = r_diff
    ys, xs = np.nonzero(w.P[0, 0] != 0)
    y, x = ys[len(ys) // 2], xs[len(xs) // 2]
    w.P[1, 2, y, x] = value
    cfg, ks = lenia.config_from_world(w)
    ctx = lenia.lenia_init(cfg, ks)
    A, P = to_dev(w.A), to_dev(w.P)
    A2, P2 = torch.empty_like(A), torch.empty_like(P)
    lenia.lenia_step(ctx, A, P, A2, P2)
    torch.cuda.synchronize()
    lenia.lenia_destroy(ctx)
    alpha = (P2.cpu().numpy() != 0).all(axis=(0, 1))
    g = oracle.diffuse(w.P[1, 2], r_diff)
    assert g[y, x] == 1.0 and alpha[_near(72, 100, y, x, r_diff + 1e-3)].any()
    np.testing.assert_allclose(P2[1, 2].cpu().numpy()[alpha], g[alpha], atol=4e-7)


BAD = [np.nan, np.inf, -np.inf, 3e38, 1e4, -2.0]


@pytest.mark.parametrize("bad", BAD)
@pytest.mark.parametrize("shape", [(300, 404, 12), (90, 100, 9), (61, 132, 6)])
def test_values_outside_the_unit_interval_stay_within_the_radius(shape, bad):
    """A value the state cannot hold reaches the potentials within R of it and no others,
    and there gives what the direct sums give."""
    H, W, R = shape
    w = inputs.single_kernel_global(H=H, W=W, R=R, patch=min(H, W) // 2)
    A = inputs.random_field(5, w.A.shape)
    clean = gpu_potentials(w, lenia.CONV_DIRECT, A)[0]
    A[0, H // 3, W // 2] = bad
    t, d = (gpu_potentials(w, p, A)[0] for p in (lenia.CONV_AUTO, lenia.CONV_DIRECT))
    far = ~_near(H, W, H // 3, W // 2, R)
    assert np.abs(t[0] - clean[0])[far].max() <= TOL_U
    np.testing.assert_array_equal(np.isfinite(t), np.isfinite(d))
    with np.errstate(invalid="ignore"):
        np.testing.assert_allclose(t, d, rtol=1e-5, atol=TOL_U)


@pytest.mark.parametrize("bad", BAD)
@pytest.mark.parametrize("kw", [dict(H=130, W=92, R=13, n_channels=3), dict(H=130, W=256, R=13, n_channels=3),
                                dict(H=105, W=100, R=9, n_channels=1)])
def test_steps_from_states_outside_the_unit_interval_equal_direct(kw, bad):
    torch = torch_mod()
    w = inputs.multi_channel(patch=40, n_geno=4, matched=True, seed_index=31, **kw)
    ys, xs = np.nonzero(w.P[0, 0] != 0)
    w.A[0, ys[len(ys) // 2], xs[len(xs) // 2]] = bad
    out = []
    for path in (lenia.CONV_AUTO, lenia.CONV_DIRECT):
        cfg, ks = lenia.config_from_world(w, path)
        ctx = lenia.lenia_init(cfg, ks)
        A, P = to_dev(w.A), to_dev(w.P)
        A2, P2 = torch.empty_like(A), torch.empty_like(P)
        lenia.lenia_step(ctx, A, P, A2, P2)
        torch.cuda.synchronize()
        out.append((A2.cpu().numpy(), P2.cpu().numpy()))
        lenia.lenia_destroy(ctx)
    np.testing.assert_array_equal(out[0][1] != 0, out[1][1] != 0)
    assert np.abs(out[0][0] - out[1][0]).max() <= 1e-5


@pytest.mark.parametrize("bad", [np.nan, np.inf, 1e38])
@pytest.mark.parametrize("shape", [(130, 140, 13, 1), (100, 72, 9, 3), (48, 60, 13, 3)])
def test_gradients_outside_the_usual_range_stay_within_the_radius(shape, bad):
    """One reversed step: the carried gradient's one bad site reaches dL/dA_0 within R."""
    torch = torch_mod()
    H, W, R, C = shape
    ks = [inputs.KernelDesc(s, d, R, inputs.KERNEL_SHELLS, (1.0,), h=0.7, mu=0.5, sigma=0.08)
          for s, d in inputs.paper_topology(C)]
    w = inputs.World(H, W, C, ks, 0.01, localized=0, maintain_genes=0)
    A0 = (0.3 + 0.4 * inputs.random_field(7, (C, H, W))).astype(np.float32)
    out = []
    for path in (lenia.CONV_AUTO, lenia.CONV_DIRECT):
        f = lenia.LeniaRollout(w, 1, conv_path=path)
        A = to_dev(A0).requires_grad_(True)
        genes = torch.from_numpy(lenia.genes_of(w)).cuda()
        g = torch.ones(A0.shape, device="cuda")
        g[0, H // 2, W // 2] = bad
        f(A, genes).backward(g)
        out.append(A.grad.cpu().numpy())
        f.close()
    np.testing.assert_array_equal(np.isfinite(out[0]), np.isfinite(out[1]))
    far = ~_near(H, W, H // 2, W // 2, R)
    assert np.abs(out[0] - out[1])[:, far].max() <= 1e-5


def test_statistics_of_a_large_world_do_not_collect_rounding():
    """A uniform world of 4096^2 sites: a thread's plain sum over its tiles would round
    alike everywhere.  Tolerance: the result's own rounding, twice."""
    torch = torch_mod()
    ks = [inputs.KernelDesc(0, 0, 4, inputs.KERNEL_SHELLS, (1.0,), h=0.5, mu=0.5, sigma=0.1),
          inputs.KernelDesc(1, 1, 4, inputs.KERNEL_SHELLS, (1.0,), h=0.5, mu=0.5, sigma=0.1)]
    w = inputs.World(4092, 4096, 2, ks, 0.0, localized=0, maintain_genes=0)
    cfg, kk = lenia.config_from_world(w)
    ctx = lenia.lenia_init(cfg, kk)
    try:
        A = torch.empty((2, 4092, 4096), device="cuda")
        out = torch.empty_like(A)
        st = torch.zeros((2, 3), device="cuda")
        for a, b in ((0.1, 0.7), (0.3, 0.9), (1.0 / 3.0, 0.6)):
            A[0], A[1] = a, b
            lenia.lenia_step(ctx, A, None, out, None, st)
            torch.cuda.synchronize()
            for c in range(2):
                exact = float(A[c, 0, 0].double()) * 4092 * 4096
                assert abs(float(st[c, 0].double()) - exact) <= 1.2e-7 * exact
    finally:
        lenia.lenia_destroy(ctx)


@pytest.mark.parametrize("n_channels", [1, 2])
@pytest.mark.parametrize("z", [1.0, 3.0])
@pytest.mark.parametrize("on_windows", [False, True])
def test_delta_sum_without_gene_maps_decides_as_the_direct_sums(n_channels, z, on_windows):
    """Global genes: E_pen of a uniform world whose sum of growths lies between the routes'."""
    k = inputs.KernelDesc(0, 0, 12, inputs.KERNEL_BUMPS, (1.0,), bump=FLAT.bump, h=1.0, mu=0.5, sigma=0.03)
    ks = [dataclasses.replace(k, src=c, dst=c) for c in range(n_channels)]
    w = inputs.World(300, 404, n_channels, ks, 0.1, localized=0, maintain_genes=0)
    w.A = np.zeros((n_channels, 300, 404), np.float32)
    mu, eps_u = _uniform_at_threshold(w, 0.03, z, on_windows)
    for k in w.kernels:
        k.mu = float(mu)
    w.eps_u = n_channels * eps_u
    a, b = _decisions(w, lenia.CONV_AUTO), _decisions(w, lenia.CONV_DIRECT)
    np.testing.assert_array_equal(a[1], b[1])


def test_delta_sum_on_fft_worlds_in_windows():
    """A power-of-two world with global genes: evolution steps (on the passes) between
    ordinary ones (in windows).  The threshold lies in the widest gap between the
    sums of two neighbouring sites, so that every route decides alike."""
    torch = torch_mod()
    w = inputs.global_multi_channel(H=256, W=128, R=13, patch=64)
    w.A = inputs.random_field(5, w.A.shape)
    for k in w.kernels:
        k.mu, k.sigma = 0.47, 0.05
    U = np.stack([oracle.potential(w.A[k.src], K) for k, K in zip(w.kernels, oracle.world_kernels(w))])
    t = np.sort(sum(k.h * np.exp(-0.5 * ((u - k.mu) / k.sigma) ** 2) for k, u in zip(w.kernels, U)).ravel())
    mid = len(t) // 2
    i = mid - 500 + int(np.argmax(np.diff(t[mid - 500:mid + 500])))
    w.eps_u = 0.5 * (t[i] + t[i + 1])
    assert t[i + 1] - t[i] > 4e-5
    _, d = _decisions(w, lenia.CONV_DIRECT)
    cfg, ks = lenia.config_from_world(w)
    ctx = lenia.lenia_init(cfg, ks)
    try:
        ev = inputs.evolution_events(w, 0, gamma_mut=0.0, gamma_pen=0.0)
        A = to_dev(w.A)
        B, E = torch.empty_like(A), torch.empty_like(A)
        ep = torch.zeros((w.height, w.width), device="cuda")
        lenia.lenia_step(ctx, A, None, B, None)
        lenia.lenia_step_evolve(ctx, A, None, E, None, ev, None, None, ep)
        lenia.lenia_step(ctx, A, None, B, None)
        torch.cuda.synchronize()
        np.testing.assert_array_equal(ep.cpu().numpy(), d)
        assert float((E - B).abs().max()) <= 1e-5
    finally:
        lenia.lenia_destroy(ctx)


@pytest.mark.parametrize("z", [1.0, 3.0])
@pytest.mark.parametrize("on_windows", [False, True])
@pytest.mark.parametrize("n_channels", [1, 2])
def test_split_step_decides_as_the_step(z, on_windows, n_channels):
    """lenia_potentials then lenia_update_from_potentials: the alpha decisions of
    lenia_step on a uniform world between the two routes' bumps."""
    torch = torch_mod()
    k = inputs.KernelDesc(0, 0, 20, inputs.KERNEL_BUMPS, (1.0,), bump=FLAT.bump, h=1.0, mu=0.5, sigma=0.03)
    ks = [dataclasses.replace(k, src=c, dst=c) for c in range(n_channels)]
    w = inputs.World(300, 404, n_channels, ks, 0.1, localized=3, maintain_genes=1)
    w.A = np.zeros((n_channels, 300, 404), np.float32)
    w.P = np.zeros((2, n_channels, 300, 404), np.float32)
    w.P[0], w.eps_u = _uniform_at_threshold(w, 0.03, z, on_windows)
    w.P[1] = np.float32(0.03)
    cfg, kk = lenia.config_from_world(w)
    ctx = lenia.lenia_init(cfg, kk)
    try:
        A, P = to_dev(w.A), to_dev(w.P)
        (A1, P1), (A2, P2) = ((torch.empty_like(A), torch.empty_like(P)) for _ in range(2))
        U = torch.empty((w.n_kernels, w.height, w.width), device="cuda")
        lenia.lenia_potentials(ctx, A, U)
        lenia.lenia_update_from_potentials(ctx, A, P, U, A1, P1)
        lenia.lenia_step(ctx, A, P, A2, P2)
        torch.cuda.synchronize()
        assert torch.equal(P1 != 0, P2 != 0)
    finally:
        lenia.lenia_destroy(ctx)


def _alone(w, n_steps):
    torch = torch_mod()
    cfg, ks = lenia.config_from_world(w)
    ctx = lenia.lenia_init(cfg, ks)
    A, P = to_dev(w.A), to_dev(w.P) if w.n_planes else None
    for _ in range(n_steps):
        A2, P2 = torch.empty_like(A), torch.empty_like(P) if w.n_planes else None
        lenia.lenia_step(ctx, A, P, A2, P2)
        A, P = A2, P2
    torch.cuda.synchronize()
    lenia.lenia_destroy(ctx)
    return A, P


@pytest.mark.parametrize("side,radii", [(64, (9, 13, 18)), (128, (9, 13, 20, 25)), (256, (9, 13)), (256, (18, 25, 13))])
@pytest.mark.parametrize("kind", ["one", "global", "local"])
@pytest.mark.parametrize("autotune", [0, 1])
def test_groups_of_worlds_equal_single_steps(side, radii, kind, autotune):
    """Grouped worlds of one size and several radii (so of several window sizes): bit for
    bit what each is on its own, and to the step's tolerance at widths of 256 k."""
    torch = torch_mod()
    ws = []
    for i, R in enumerate(radii):
        if kind == "one":
            w = inputs.single_kernel_global(H=side, W=side, R=R, patch=side // 2, sigma=0.05, mu=0.42)
            w.A = inputs.random_field(100 * side + i, w.A.shape)
        elif kind == "global":
            w = inputs.global_multi_channel(H=side, W=side, R=R, patch=side // 2)
            w.A = inputs.random_field(100 * side + i, w.A.shape)
        else:
            w = inputs.multi_channel(H=side, W=side, R=R, patch=side // 4, n_geno=3, matched=True, seed_index=60 + i)
        ws.append(w)
    if kind != "one":        # one topology and one set of global genes, so that they group
        for w in ws[1:]:
            for k, k0 in zip(w.kernels, ws[0].kernels):
                k.h, k.mu, k.sigma = k0.h, k0.mu, k0.sigma
    b = lenia.lenia_batch_init(ws, autotune=bool(autotune))
    try:
        assert all(lenia.lenia_batch_group_of(b, i) == 0 for i in range(len(ws)))
        A = [to_dev(w.A) for w in ws]
        P = [to_dev(w.P) if w.n_planes else None for w in ws]
        lenia.lenia_batch_rollout(b, A, P, 3)
        lenia.lenia_batch_check(b)
        for i, w in enumerate(ws):
            A1, P1 = _alone(w, 3)
            if side % 256:
                assert torch.equal(A[i], A1) and (P1 is None or torch.equal(P[i], P1))
            assert float((A[i] - A1).abs().max()) <= 3e-5
    finally:
        lenia.lenia_batch_destroy(b)


@pytest.mark.parametrize("side,n_kernels,route", [(64, 4, lenia.ROUTE_BLOCK), (128, 1, lenia.ROUTE_BLOCK),
                                                  (128, 4, lenia.ROUTE_STEPS), (64, 5, lenia.ROUTE_STEPS)])
def test_small_one_channel_worlds_step_as_they_roll(side, n_kernels, route):
    """Steps with statistics, potentials and rollouts of 2 to 6 steps of the worlds around
    the one-block rollout's limits, against the oracle's steps."""
    torch = torch_mod()
    w = inputs.single_kernel_global(H=side, W=side, R=13, patch=side, sigma=0.2, mu=0.42)
    w.kernels = [inputs.KernelDesc(0, 0, 13 - i, inputs.KERNEL_SHELLS, (1.0,), h=1.0 - 0.15 * i, mu=0.42 + 0.02 * i,
                                   sigma=0.2 + 0.01 * i) for i in range(n_kernels)]
    w.dt = 0.02
    # a step passes an error on by at most L, the steepest growth's share
    L = 1 + w.dt * sum(2 * k.h * np.exp(-0.5) / k.sigma for k in w.kernels)
    tol = lambda n: 1e-5 * (L**n - 1) / (L - 1)
    U = gpu_potentials(w)[0]
    ref = np.stack([oracle.potential(w.A[k.src], K) for k, K in zip(w.kernels, oracle.world_kernels(w))])
    assert np.abs(U - ref).max() <= TOL_U
    cfg, ks = lenia.config_from_world(w)
    ctx = lenia.lenia_init(cfg, ks)
    try:
        assert lenia.lenia_rollout_route(ctx) == route
        for n in (2, 3, 6):
            A, st = to_dev(w.A), torch.zeros((n, 1, 3), device="cuda")
            B = A.clone()
            lenia.lenia_rollout(ctx, A, None, n)
            lenia.lenia_rollout(ctx, B, None, n, st)
            torch.cuda.synchronize()
            want = oracle.rollout(w, n)[0]
            assert np.abs(A.cpu().numpy() - want).max() <= tol(n)
            assert np.abs(B.cpu().numpy() - want).max() <= tol(n)
            # (the mass: a nearly even world has no well-defined centre)
            np.testing.assert_allclose(st[n - 1, :, 0].cpu().numpy(), oracle.stats(B.cpu().numpy())[:, 0], rtol=1e-5)
    finally:
        lenia.lenia_destroy(ctx)


@pytest.mark.parametrize("autotune", [0, 1])
def test_ring_worlds_in_a_batch(autotune):
    """The batch's second state holds a ring world's kernel genes too (nine planes a
    kernel): bit for bit the steps of the world on its own."""
    torch = torch_mod()
    ws = [inputs.ring_world(H=64, W=64, R=6, n_rings=12, patch=24, n_geno=2) for _ in range(2)]
    ws.append(inputs.single_kernel_global(H=64, W=64, R=9, patch=32))
    b = lenia.lenia_batch_init(ws, autotune=bool(autotune), conv_path=lenia.CONV_AUTO)
    try:
        A = [to_dev(w.A) for w in ws]
        P = [to_dev(w.P) if w.n_planes else None for w in ws]
        lenia.lenia_batch_rollout(b, A, P, 3)
        lenia.lenia_batch_check(b)
        for i in (0, 1):
            cfg, ks = lenia.config_from_world(ws[i], lenia.lenia_batch_conv_path(b, i))
            ctx = lenia.lenia_init(cfg, ks)
            A1, P1 = to_dev(ws[i].A), to_dev(ws[i].P)
            for _ in range(3):
                A2, P2 = torch.empty_like(A1), torch.empty_like(P1)
                lenia.lenia_step(ctx, A1, P1, A2, P2)
                A1, P1 = A2, P2
            torch.cuda.synchronize()
            lenia.lenia_destroy(ctx)
            assert torch.equal(A[i], A1) and torch.equal(P[i], P1)
    finally:
        lenia.lenia_batch_destroy(b)


@pytest.mark.parametrize("kw", [dict(H=64, W=64, R=6, n_rings=12), dict(H=128, W=128, R=12, n_rings=24, n_channels=1),
                                dict(H=256, W=128, R=9, n_rings=4)])
def test_ring_worlds_without_maintenance_in_windows(kw):
    """Power-of-two ring worlds whose genes are not maintained may convolve their rings in
    windows: ring potentials against the oracle (unnormalised sums of up to 50
    values), and a step (its genes unchanged)."""
    torch = torch_mod()
    w = inputs.ring_world(patch=24, n_geno=2, **kw)
    w.maintain_genes = 0
    cfg, ks = lenia.config_from_world(w)
    ctx = lenia.lenia_init(cfg, ks)
    try:
        A, P = to_dev(w.A), to_dev(w.P)
        V = torch.empty((w.n_channels, w.n_rings, w.height, w.width), device="cuda")
        lenia.lenia_potentials(ctx, A, V)
        A2, P2 = torch.empty_like(A), torch.empty_like(P)
        lenia.lenia_step(ctx, A, P, A2, P2)
        torch.cuda.synchronize()
        rings = np.stack([oracle.ring_potentials(w.A[c], w.kernels[0].radius, w.n_rings) for c in range(w.n_channels)])
        assert np.abs(V.cpu().numpy() - rings).max() <= 2e-5
        want = oracle.ring_step(w)[0]
        assert np.abs(A2.cpu().numpy() - want).max() <= 1e-5 and torch.equal(P2, P)
    finally:
        lenia.lenia_destroy(ctx)


@pytest.mark.parametrize("sigma", [1e-40, 1e-37, 1e-30])
def test_one_block_rollouts_of_vanishing_bumps(sigma):
    """A sigma whose reciprocal is infinite: rollouts give what steps give."""
    torch = torch_mod()
    w = inputs.single_kernel_global(H=64, W=64, R=9, patch=32, sigma=0.05, mu=0.3)
    w.kernels[0].sigma = float(np.float32(sigma))
    cfg, ks = lenia.config_from_world(w)
    ctx = lenia.lenia_init(cfg, ks)
    try:
        A = to_dev(w.A)
        S = A.clone()
        lenia.lenia_rollout(ctx, A, None, 3)
        for _ in range(3):
            T = torch.empty_like(S)
            lenia.lenia_step(ctx, S, None, T, None)
            S = T
        torch.cuda.synchronize()
        assert float((A - S).abs().max()) <= 3e-5
    finally:
        lenia.lenia_destroy(ctx)

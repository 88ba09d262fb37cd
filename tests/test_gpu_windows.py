"""The convolution in overlapping spectral windows and the per-site update
kernel: potentials, steps, alpha decisions and gradients at the sizes where the
windows' geometry changes (worlds smaller than a window, one window wide,
ragged last windows, odd radii) against the FP64 oracle and the direct sums.
GPU only."""
import numpy as np
import pytest

import oracle
from paper_2304_05639_gb300 import build, inputs, lenia
from gpu_util import TOL_STEP, TOL_U, alpha_margin, compare_step, gpu_potentials, gpu_step, to_dev, torch_mod

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    build.build()
    oracle.build()
    torch_mod()


def _oracle_u(w):
    ks = oracle.world_kernels(w)
    return np.stack([oracle.potential(w.A[k.src], K) for k, K in zip(w.kernels, ks)])


# (H, W, R, channels): smaller than the window, exactly one window (64, 128)
# in one or both axes, a last window of 4 columns or 1 row, odd and even radii
SHAPES = [(48, 60, 15, 1), (64, 64, 13, 1), (64, 100, 9, 1), (128, 128, 20, 3), (61, 132, 7, 1), (105, 104, 12, 2),
          (300, 404, 12, 1), (257, 92, 18, 3), (90, 128, 25, 1), (41, 44, 20, 1)]


def _global(H, W, R, C):
    if C == 1:
        w = inputs.single_kernel_global(H=H, W=W, R=R, patch=min(H, W) // 2)
    else:
        w = inputs.global_multi_channel(H=H, W=W, R=R, patch=min(H, W) // 2, n_channels=C)
    w.A = inputs.random_field(H * 1000 + W, w.A.shape)
    return w


@pytest.mark.parametrize("shape", SHAPES)
def test_window_potentials_match_oracle(shape):
    w = _global(*shape)
    U, _ = gpu_potentials(w)
    err = np.abs(U - _oracle_u(w)).max()
    print(shape, "max |dU|", err)
    assert err <= TOL_U


# grids below and above two blocks an SM, where a block's thread count changes
@pytest.mark.parametrize("shape", [(900, 800, 5, 1), (1000, 1100, 5, 1), (300, 560, 20, 3), (600, 560, 20, 3)])
def test_window_potentials_of_larger_grids_match_oracle(shape):
    w = _global(*shape)
    U, _ = gpu_potentials(w)
    err = np.abs(U - _oracle_u(w)).max()
    print(shape, "max |dU|", err)
    assert err <= TOL_U


@pytest.mark.parametrize("shape", SHAPES[2:8])
def test_unaligned_state_equals_aligned(shape):
    """A caller's A that starts 4 bytes past an 8-byte boundary takes scalar loads: same bits."""
    torch = torch_mod()
    w = _global(*shape)
    cfg, ks = lenia.config_from_world(w)
    ctx = lenia.lenia_init(cfg, ks)
    try:
        A = to_dev(w.A)
        flat = torch.empty(A.numel() + 1, device="cuda")
        B = flat[1:].view_as(A)
        B.copy_(A)
        U, V = (torch.empty((w.n_kernels, w.height, w.width), device="cuda") for _ in range(2))
        lenia.lenia_potentials(ctx, A, U)
        lenia.lenia_potentials(ctx, B, V)
        torch.cuda.synchronize()
        assert torch.equal(U, V)
    finally:
        lenia.lenia_destroy(ctx)


LOCAL = [dict(H=72, W=100, R=9, n_channels=1), dict(H=130, W=92, R=13, n_channels=3), dict(H=105, W=256, R=12, n_channels=2),
         dict(H=96, W=80, R=7, n_channels=4)]
ALL3 = inputs.LOC_MU | inputs.LOC_SIGMA | inputs.LOC_H


@pytest.mark.parametrize("kw", LOCAL)
@pytest.mark.parametrize("variant", [dict(), dict(r_diff=2), dict(localized=ALL3), dict(localized=ALL3, r_diff=2),
                                     dict(alpha_on=1), dict(growth_form=1)])
def test_site_kernel_step_matches_oracle_and_direct(kw, variant):
    """One step of ragged worlds of 1 to 4 channels (3 to 24 kernels) against the
    oracle; and the decisions equal those of the direct sums at every site."""
    variant = dict(variant)
    w = inputs.multi_channel(patch=40, n_geno=4, matched=True, localized=variant.pop("localized", 3), seed_index=31, **kw)
    for k, v in variant.items():
        setattr(w, k, v)
    g = gpu_step(w, stats=True)
    A1, P1, U, al = oracle.step(w, return_u=True, return_alpha=True)
    Ph = np.stack([[oracle.diffuse(w.P[p, k], w.r_diff) for k in range(w.n_kernels)] for p in range(w.n_planes)])
    print(kw, variant, compare_step(w, g, A1, P1, al, alpha_margin(w, U, Ph), min_alpha1=0))
    np.testing.assert_allclose(g["stats"], oracle.stats(g["A"]), rtol=1e-5)
    d = gpu_step(w, lenia.CONV_DIRECT)
    np.testing.assert_array_equal(g["P"] != 0, d["P"] != 0)
    assert np.abs(g["A"] - d["A"]).max() <= TOL_STEP


@pytest.mark.parametrize("eps_u", [0.01, 0.3, 0.55])
def test_many_near_threshold_decisions_equal_direct(eps_u):
    """A world whose growth passes the threshold almost everywhere (uniform genes on
    noise, eps_u inside the bump's range): every alpha and Delta_sum decision is
    that of the direct sums, also where windows and sums round to either side."""
    torch = torch_mod()
    H, W = 210, 300
    w = inputs.localized_single_channel(H=H, W=W, R=9, patch=64, n_geno=6, live=True)
    w.P[0], w.P[1] = 0.47, 0.02
    w.A = inputs.random_field(5, w.A.shape)
    w.eps_u = eps_u
    ev = inputs.evolution_events(w, 0, gamma_mut=0.0, gamma_pen=0.0)
    res = []
    for path in (lenia.CONV_AUTO, lenia.CONV_DIRECT):
        cfg, ks = lenia.config_from_world(w, path)
        ctx = lenia.lenia_init(cfg, ks)
        try:
            A, P = to_dev(w.A), to_dev(w.P)
            A2, P2 = torch.empty_like(A), torch.empty_like(P)
            al = torch.zeros((H, W), dtype=torch.uint8, device="cuda")
            ep = torch.zeros((H, W), dtype=torch.float32, device="cuda")
            lenia.lenia_step_evolve(ctx, A, P, A2, P2, ev, None, al, ep)
            torch.cuda.synchronize()
            res.append((al.cpu().numpy(), ep.cpu().numpy()))
        finally:
            lenia.lenia_destroy(ctx)
    assert 0.02 < res[0][0].mean() < 0.98
    np.testing.assert_array_equal(res[0][0], res[1][0])
    np.testing.assert_array_equal(res[0][1], res[1][1])


@pytest.mark.parametrize("shape", [(48, 60, 13, 1), (100, 72, 9, 3), (130, 140, 13, 3)])
def test_window_gradients_match_direct(shape):
    """dL/dA_0 and the gene gradients of a three-step rollout through the windows'
    transposed convolution equal the direct route's (relative 2-norm 1e-4: the
    two round their potentials differently, at most 2e-6 per step)."""
    torch = torch_mod()
    w = _global(*shape)
    out = []
    for path in (lenia.CONV_AUTO, lenia.CONV_DIRECT):
        f = lenia.LeniaRollout(w, 3, ckpt_every=2, conv_path=path)
        A = to_dev(w.A).requires_grad_(True)
        genes = torch.from_numpy(lenia.genes_of(w)).cuda()
        genes[:, 1] = 0.08
        genes.requires_grad_(True)
        gen = torch.Generator().manual_seed(3)
        f(A, genes).backward(torch.randn(A.shape, generator=gen).cuda())
        out.append((A.grad.double(), genes.grad.double()))
        f.close()
    for a, b in zip(*out):
        assert float((a - b).norm()) <= 1e-4 * float(b.norm())


@pytest.mark.parametrize("side,n_kernels,form", [(64, 1, 0), (64, 2, 1), (64, 4, 0), (128, 1, 1), (128, 3, 0)])
def test_one_block_rollout_matches_oracle_and_steps(side, n_kernels, form):
    """Whole rollouts in one block: 2 steps against the oracle and 7 against
    repeated single steps, aligned and 4 bytes past a 16-byte boundary."""
    torch = torch_mod()
    w = inputs.single_kernel_global(H=side, W=side, R=13, patch=side, sigma=0.05, mu=0.42)
    w.kernels = [inputs.KernelDesc(0, 0, 13 - 2 * i, inputs.KERNEL_SHELLS, (1.0, 0.5)[:1 + i % 2], h=1.0 - 0.2 * i,
                                   mu=0.42 + 0.02 * i, sigma=0.05 + 0.01 * i) for i in range(n_kernels)]
    w.growth_form = form
    cfg, ks = lenia.config_from_world(w)
    ctx = lenia.lenia_init(cfg, ks)
    try:
        assert lenia.lenia_rollout_route(ctx) == lenia.ROUTE_BLOCK
        A = to_dev(w.A)
        lenia.lenia_rollout(ctx, A, None, 2)
        ref = oracle.rollout(w, 2)[0]
        assert np.abs(A.cpu().numpy() - ref).max() <= 2 * TOL_STEP
        S, B = to_dev(w.A), to_dev(w.A)
        for _ in range(7):
            T = torch.empty_like(S)
            lenia.lenia_step(ctx, S, None, T, None)
            S = T
        lenia.lenia_rollout(ctx, B, None, 7)
        flat = torch.empty(S.numel() + 1, device="cuda")
        D = flat[1:].view_as(S)
        D.copy_(to_dev(w.A))
        lenia.lenia_rollout(ctx, D, None, 7)
        torch.cuda.synchronize()
        assert torch.equal(B, D)
        assert float((S - B).abs().max()) <= 7 * TOL_STEP
    finally:
        lenia.lenia_destroy(ctx)

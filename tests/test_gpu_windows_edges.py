"""The windows and the per-site update kernel off the usual worlds: channels that
no kernel reads, narrow bumps and large radii (every alpha decision is that of
the direct sums), values outside [0, 1], infinite genes, long sums, and groups
of worlds.  GPU only."""
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


@pytest.mark.parametrize("shape,topology", [((100, 72, 9), [(0, 1)]), ((64, 64, 9), [(0, 1)]), ((130, 140, 13), [(0, 0), (0, 1)]),
                                            ((300, 404, 12), [(1, 0), (1, 2), (1, 1)]), ((128, 128, 20), [(2, 0)])])
def test_gradient_of_channels_that_no_kernel_reads(shape, topology):
    """dL/dA_0 of a channel that is only written is the carried gradient itself: the
    windows' transposed convolution equals the direct route's (relative 2-norm
    1e-4 per channel, as test_window_gradients_match_direct)."""
    H, W, R = shape
    C = max(max(t) for t in topology) + 1
    ks = [inputs.KernelDesc(s, d, R, inputs.KERNEL_SHELLS, (1.0,), h=0.7, mu=0.5, sigma=0.08) for s, d in topology]
    w = inputs.World(H, W, C, ks, 0.1, localized=0, maintain_genes=0)
    w.A = inputs.random_field(H + W, (C, H, W))
    (a, ga), (b, gb) = (_gradients(w, 3, p) for p in (lenia.CONV_AUTO, lenia.CONV_DIRECT))
    for c in range(C):
        assert float((a[c] - b[c]).norm()) <= 1e-4 * float(b[c].norm())
    assert float((ga - gb).norm()) <= 1e-4 * float(gb.norm())

"""Sides whose rows are cut into segments of less than 128 pixels, or of two
widths, with more work units than resident CTAs, so that CTAs go from narrow
units to wide ones: every chain must come out as it does alone."""
import numpy as np
import pytest
import torch

import paper_1906_06297_gb300 as ising

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    ising.build()


def setup(L, C, seed):
    mv = ising.BlockMove(L, C, 0.4406868)
    mv.batch.init(ising.ISING_INIT_RANDOM, seed)
    mv.batch.run(5, seed)
    torch.cuda.synchronize()
    th = np.random.default_rng(seed).normal(0.0, 0.2, ising.ising_net_param_count()).astype(np.float32)
    return mv, torch.from_numpy(th).cuda(), (L // 8) ** 2


# segments: 96 + 64, 128 + 96, 96 + 96, 64, 32
@pytest.mark.parametrize("L,C", [(160, 90), (224, 50), (192, 40), (64, 200), (32, 400)])
def test_many_chains_equal_single_chains(L, C):
    mv, params, nb = setup(L, C, 3)
    logits = torch.zeros((C, nb), dtype=torch.float32, device="cuda")
    ising.ising_net_forward(L, C, mv.black, mv.white, None, params, logits, mv.work)
    plane = L * L // 4
    one = torch.zeros((1, nb), dtype=torch.float32, device="cuda")
    for c in (0, 1, C // 2, C - 1):
        ising.ising_net_forward(L, 1, mv.black[c * plane:(c + 1) * plane], mv.white[c * plane:(c + 1) * plane], None, params,
                                one, mv.work)
        ising.ising_net_check()
        assert torch.equal(one[0], logits[c])


@pytest.mark.parametrize("L,C", [(160, 90), (224, 50), (96, 120)])
def test_gradient_of_copies_is_a_multiple(L, C):
    """C copies of one chain with the same dlogits: C times its gradient, up to
    the rounding of FP32 sums (C n_pixels terms in a few thousand partials:
    1e-5 of each layer's largest value is several times their error)."""
    mv, params, nb = setup(L, 1, 7)
    black, white = mv.black.repeat(C), mv.white.repeat(C)
    work = torch.empty(ising.ising_net_workspace_bytes(L, C, True), dtype=torch.uint8, device="cuda")
    d = torch.from_numpy(np.random.default_rng(1).normal(0.0, 1.0, (1, nb)).astype(np.float32)).cuda()
    grads = []
    for n, b, w in ((1, mv.black, mv.white), (C, black, white)):
        logits = torch.zeros((n, nb), dtype=torch.float32, device="cuda")
        g = torch.zeros_like(params)
        ising.ising_net_forward(L, n, b, w, None, params, logits, work, train=True)
        ising.ising_net_backward(L, n, b, w, params, d.repeat(n, 1), g, work)
        ising.ising_net_check()
        grads.append(g.double().cpu().numpy())
    o = 0
    for size in (288, 32, 9216, 32, 9216, 32, 288, 1):
        a, b = C * grads[0][o:o + size], grads[1][o:o + size]
        assert np.abs(a - b).max() <= 1e-5 * np.abs(a).max()
        o += size

"""Weight gradients of the 32 -> 32 layers on sides that are no multiple of 128 are
FP32 sums of the unrounded output gradients.  The parameters are chosen so that
activations and output gradients are known exactly: saturated GELUs (gelu(z) = z and
gelu'(z) = 1 from z = 16 on) make every a1, a2 a small whole number and every dz3, dz2
the same 24-bit number v, of which two bfloat16 parts leave 2^-18 behind."""
import numpy as np
import pytest
import torch

import paper_1906_06297_gb300 as ising

pytestmark = pytest.mark.gpu
CH = 32
V = 1 + 2.0**-9 - 2.0**-18 - 2.0**-23


@pytest.fixture(scope="module", autouse=True)
def built():
    ising.build()


@pytest.mark.parametrize("L,C", [(32, 1), (96, 1), (160, 1)])
def test_weight_gradients_see_every_bit_of_the_output_gradient(L, C):
    a = 16.0 + np.arange(CH)
    W3 = np.zeros((CH, CH, 9))
    for i in range(CH):  # dz2 = dz3 (1 + 2^-9 - 2^-18 - 2^-23), from a dz3 that rounds to 1
        W3[i, i, [4, 0, 8]] = 1.0, 2.0**-9, -(2.0**-18 + 2.0**-23)
    W4 = np.zeros((CH, 9))
    W4[:, 4] = 1.0
    theta = np.concatenate([np.zeros(CH * 9), a, np.zeros(CH * CH * 9), a, W3.ravel(), np.full(CH, 16.0), W4.ravel(), [0.0]])
    params = torch.from_numpy(theta.astype(np.float32)).cuda()
    mv = ising.BlockMove(L, C, 0.44)
    mv.batch.init(ising.ISING_INIT_RANDOM, 1)
    nb = (L // 8) ** 2
    logits = torch.zeros((C, nb), dtype=torch.float32, device="cuda")
    d = torch.full((C, nb), 64 * V, dtype=torch.float32, device="cuda")
    assert float(d[0, 0]) == 64 * V
    work = torch.empty(ising.ising_net_workspace_bytes(L, C, True), dtype=torch.uint8, device="cuda")
    grad = torch.zeros_like(params)
    ising.ising_net_forward(L, C, mv.black, mv.white, None, params, logits, work, train=True)
    ising.ising_net_backward(L, C, mv.black, mv.white, params, d, grad, work)
    ising.ising_net_check()
    g = grad.cpu().numpy().astype(np.float64)
    n = C * L * L
    # A row segment's sum takes a truncated addition per 16 pixels and as much again for
    # the products' own alignment, 2^-23 each at most; its CTA adds up to three such rows,
    # 8 warps of the reduction an eighth of the CTAs each, and their sums, half that each.
    # (A bias takes 4 pixels per lane and row, three shuffles and four warps.)
    segs = -(-L // 128)
    tw = -(-L // 32 // segs) * 32
    ctas = min(152, C * segs * L)
    tol = (2 * tw / 16 + 0.5 * (3 + ctas / 8 + 8)) * 2.0**-23
    assert tol < 0.9 * 2.0**-18  # less than what two parts would miss
    o = 0
    for size, want in ((CH * 9, None), (CH, None), (CH * CH * 9, n * V * a[None, :, None]), (CH, n * V),
                       (CH * CH * 9, n * V * a[None, :, None]), (CH, n * V)):
        if want is not None:
            got = g[o:o + size].reshape((CH, CH, 9) if size > CH else CH)
            assert np.abs(got / want - 1).max() <= tol
        o += size

"""The training gradient's sums across CTAs where their last bits show.  With every parameter
0 the network's outputs are 0, so the gradient of output bias c is -2 / (3 n) times the sum of
the targets t_c.  The targets here need 53 bits together and cancel but for the smallest: every
sum of them in doubles is exact, in any order.  And sums beyond a float's range whose mean is
within it."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def gpu():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2105_12912_gb300 import api
    return api


@pytest.mark.parametrize("order", [0, 1, 2])
@pytest.mark.parametrize("scale", [0, -140])
def test_bias_gradient_in_53_bits(gpu, order, scale):
    n = 30000
    vals = np.array([2.0 ** 51, 2.0 ** 25, 0.5, -(2.0 ** 51), -(2.0 ** 25)]) * 2.0 ** (scale / 2)
    vals = vals[np.random.default_rng(order).permutation(5)]
    tgt = np.zeros((n, 3))
    for i, v in enumerate(vals):
        tgt[12 * (7 + 20 * i) + order, 1] = v  # rows far apart: different CTAs
    tgt32 = tgt.astype(np.float32)
    assert np.array_equal(tgt32.astype(np.float64), tgt)
    w = torch.zeros(gpu.MLP_PARAMS, device="cuda")
    _, g = gpu.selector_grad(w, torch.ones((n, 8), device="cuda"), torch.from_numpy(tgt32).cuda())
    g = g.cpu().numpy()
    want = np.zeros(gpu.MLP_PARAMS)
    want[-2] = -2.0 * tgt[:, 1].sum() / (3.0 * n)
    assert want[-2] != 0.0
    # (the scale 1 / 3n is one rounded double: at most one unit of the float)
    assert abs(float(g[-2]) - want[-2]) <= 2.0 ** -23 * abs(want[-2])
    assert not np.delete(g, gpu.MLP_PARAMS - 2).any()


def test_sums_beyond_a_float(gpu):
    n = 30000
    tgt = torch.full((n, 3), 1e35, device="cuda")
    _, g = gpu.selector_grad(torch.zeros(gpu.MLP_PARAMS, device="cuda"), torch.ones((n, 8), device="cuda"), tgt)
    want = -2.0 * float(tgt[0, 0]) / 3.0  # (each CTA's 197 rows sum to 4e37, all of them to 6e39)
    assert ((g[-3:].double() - want).abs() <= 1e-5 * abs(want)).all()

"""The training gradient at the edges of its row loop: row counts around a warp's pairs, its
ballots of 32 rows and the launch's warps, and rows that take no part -- none, some, all, and
with values no number may come from.

Tolerance: the FP32 gradient within 1e-4 of the oracle's double-precision one, relative to
its largest entry, and the loss within 1e-5, as for whole fields (sums of a few thousand
terms in FP32 lose about sqrt(n) 2^-24)."""
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


@pytest.mark.parametrize("keep", ["all", "alternate", "one", "third"])
@pytest.mark.parametrize("n", [1, 2, 3, 31, 32, 33, 64, 65, 1823, 1825, 60001])
def test_gradient_rows(gpu, orc, n, keep):
    rng = np.random.default_rng(n)
    w = (rng.standard_normal(gpu.MLP_PARAMS) * 0.3).astype(np.float32)
    feat = rng.standard_normal((n, 8)).astype(np.float32)
    # (targets off zero: the sums do not cancel, and one unit at its kink weighs 1 / n)
    tgt = (3.0 + rng.standard_normal((n, 3))).astype(np.float32)
    i = np.arange(n)
    valid = {"all": i >= 0, "alternate": i % 2 == 0, "one": i == n - 1, "third": i % 3 == 1}[keep]
    feat[~valid] = np.nan  # rows that take no part
    tgt[~valid] = np.inf
    loss, g = gpu.selector_grad(torch.from_numpy(w).cuda(), torch.from_numpy(feat).cuda(), torch.from_numpy(tgt).cuda(),
                                torch.from_numpy(valid.astype(np.uint8)).cuda())
    g = g.cpu().numpy()
    if not valid.any():
        assert loss == 0.0 and not g.any()
        return
    ref_loss, ref_g = orc.mlp_loss_grad(w, feat[valid], tgt[valid])
    assert abs(loss - ref_loss) <= 1e-5 * max(1.0, abs(ref_loss))
    assert np.abs(g - ref_g).max() <= 1e-4 * np.abs(ref_g).max()

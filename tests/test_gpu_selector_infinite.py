"""The training gradient where activations overflow: with positive parameters and inputs that
overflow the first layer every entry is an infinity, never a NaN, whatever the row count (a
warp takes its rows in pairs, the last one alone)."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def gpu():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2105_12912_gb300 import api
    return api


@pytest.mark.parametrize("n", [1, 2, 3, 33, 1824, 1825, 40000])
def test_infinite_activations(gpu, n):
    w = torch.full((gpu.MLP_PARAMS,), 0.5, device="cuda")
    feat = torch.full((n, 8), 3e38, device="cuda")
    loss, g = gpu.selector_grad(w, feat, torch.zeros((n, 3), device="cuda"))
    assert loss == float("inf")
    assert torch.isposinf(g).all()

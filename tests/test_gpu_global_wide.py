"""GPU parity of the global reconstruction on fields much wider than they have rows, and on
fields thinner than a block: one and more turns of the row-sum scan with either CTA size, the
shapes on both sides of the line between the scans and of the rows the last pass takes.

Archives and reconstructions must equal the oracle's byte for byte (no tolerance)."""
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


@pytest.mark.parametrize("shape", [
    (16, 70000),                # one turn, CTAs of 1024
    (1, 600000),                # 9375 blocks: two turns of 8192
    (400, 8400),                # more rows than two an SM: CTAs of 256
    (5, 61, 32790),             # 2050 blocks: two turns of 2048
    (4, 4096), (4, 4097),       # 64 blocks and 65: a thread per row, a CTA per row
    (1, 3, 1024), (1, 3, 1025), (81, 4160), (81, 4161),
    (30, 255), (30, 256), (65, 257), (9, 300), (17, 1000),
    (2, 700, 40), (15, 20, 20), (3, 5, 40000), (48, 3, 1), (49, 1),
])
def test_wide_and_thin(gpu, orc, shape):
    x = np.random.default_rng(sum(shape)).standard_normal(shape).astype(np.float32)
    for ax in range(len(shape)):
        x = np.cumsum(x, axis=ax).astype(np.float32)
    x[..., shape[-1] // 2: shape[-1] // 2 + shape[-1] // 5] = 0.0
    ar, nb, st = gpu.compress(torch.from_numpy(x).cuda(), 0.5, "abs", radius=12, global_lorenzo=True)
    ost, ref = orc.compress_ex(x, orc.EB_ABS, 0.5, radius=12, select=gpu.SELECT["exhaustive"], global_lorenzo=True)
    assert st == ost == 0
    assert nb == ref.size and np.array_equal(ar[:nb].cpu().numpy(), ref)
    buf = torch.zeros(x.size + 1, dtype=torch.float32, device="cuda")
    y, _ = gpu.decompress(ar, nb, out=buf[1:].view(x.shape))
    _, yr = orc.decompress(ref, x.size)
    assert np.array_equal(y.cpu().numpy().ravel().view(np.uint32), yr.view(np.uint32))

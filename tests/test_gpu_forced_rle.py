"""GPU parity of forced run-length coding, whose blocks have launches of their own: run counts
from one a block to one an element (odd counts among them), groups of 256 blocks before a
block's place, cut blocks, many outlier records, double fields, global prediction, and an
archive buffer one byte short.

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


@pytest.mark.parametrize("kind", ["f32", "f64", "global"])
@pytest.mark.parametrize("scale", [0.0, 0.02, 1.0])
@pytest.mark.parametrize("shape", [(1,), (4095,), (4097,), (4096 * 513 + 7,), (65, 130), (1100, 1030), (17, 33, 50)])
def test_forced_rle(gpu, orc, shape, scale, kind):
    rng = np.random.default_rng(sum(shape))
    x = (scale * rng.standard_normal(shape)).cumsum(axis=-1)
    x[..., : shape[-1] // 4] = 0.25
    x = x.astype(np.float64 if kind == "f64" else np.float32)
    xd = torch.from_numpy(np.ascontiguousarray(x)).cuda()
    kw = {"global_lorenzo": True} if kind == "global" else {}
    ar, nb, st = gpu.compress(xd, 0.01, "abs", radius=20, select="rle", **kw)
    compress = orc.compress_f64 if kind == "f64" else orc.compress_ex
    ost, ref = compress(x, orc.EB_ABS, 0.01, radius=20, select=orc.SEL_RLE, **kw)
    assert st == ost == 0
    assert nb == ref.size and np.array_equal(ar[:nb].cpu().numpy(), ref)
    short = torch.full((nb + 256,), 0xa5, dtype=torch.uint8, device="cuda")
    _, _, st = gpu.compress(xd, 0.01, "abs", radius=20, select="rle", out=short[:nb - 1], raise_on_error=False, **kw)
    assert st == 5 and bool((short[nb - 1:] == 0xa5).all())  # CSZ_E_CAPACITY
    y, _ = gpu.decompress(ar, nb)
    assert float((y.double() - xd.double()).abs().max()) <= 0.01

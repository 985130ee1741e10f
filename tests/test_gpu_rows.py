"""GPU parity of the row-wise paths at their edges: 3-D blocks cut by the field's faces
(chunked and global prediction, FP32), and the global reconstruction's row sums, strips and
ragged rows in one, two and three dimensions -- with many outliers, verbatim patches, and
runs, in cut blocks and in whole ones.

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


def _field(orc, shape, kind, eb):
    n = int(np.prod(shape))
    rng = np.random.default_rng(n)
    x = rng.standard_normal(shape).astype(np.float32)
    if kind == "patches":
        # half points of the quantization step at large |k|: the neighbours of a half point
        # meet the bound on one side only, or not at all
        _, _, _, x2, _ = orc.eb_params(orc.EB_ABS, eb)
        vals = []
        for k in [1, 3, 1000, 654321, 3000000, 7000000]:
            c = np.float32((k + 0.5) * float(x2))
            for v in (np.nextafter(c, np.float32(0)), c, np.nextafter(c, np.float32(np.inf))):
                vals += [v, -v]
        return np.resize(np.array(vals, dtype=np.float32), n).reshape(shape)
    for ax in range(len(shape)):
        x = np.cumsum(x, axis=ax).astype(np.float32)
    if kind == "runs":
        x[tuple(slice(s // 4, None) for s in shape)] = 0.0
    return x


@pytest.mark.parametrize("global_lorenzo", [False, True])
@pytest.mark.parametrize("kind", ["outliers", "patches", "runs"])
@pytest.mark.parametrize("shape", [(16, 16, 16), (17, 33, 15), (5, 3, 2), (40, 144, 1), (1, 1, 100), (33, 160, 52),
                                   (200, 1, 3), (64, 64), (65, 130), (700, 3), (3, 700), (4096,), (9001,)])
def test_rows_parity(gpu, orc, shape, kind, global_lorenzo):
    eb = 0.0123456789 if kind == "patches" else 0.5
    radius = 6 if kind == "outliers" else 512
    x = _field(orc, shape, kind, eb)
    xd = torch.from_numpy(np.ascontiguousarray(x)).cuda()
    ar, nb, st = gpu.compress(xd, eb, "abs", radius=radius, global_lorenzo=global_lorenzo, raise_on_error=False)
    ost, ref = orc.compress_ex(x, orc.EB_ABS, eb, radius=radius, select=gpu.SELECT["exhaustive"],
                               global_lorenzo=global_lorenzo, raise_on_error=False)
    assert st == ost == 0
    assert nb == ref.size and np.array_equal(ar[:nb].cpu().numpy(), ref)
    # an output that starts off a 16-byte boundary, as a slice of a larger buffer may
    buf = torch.zeros(x.size + 1, dtype=torch.float32, device="cuda")
    y, _ = gpu.decompress(ar, nb, out=buf[1:].view(x.shape))
    _, yr = orc.decompress(ref, x.size)
    assert np.array_equal(y.cpu().numpy().ravel().view(np.uint32), yr.view(np.uint32))

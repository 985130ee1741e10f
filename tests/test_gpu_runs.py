"""GPU parity of run blocks at the edges of the run expansion: one run a block, as many runs
as a pass of the CTA takes and one more, a run per element, runs that end on word and
thread boundaries; whole and cut blocks of every dimensionality, FP32 and double, single
fields and a batch of mixed dimensionality.

Archives and reconstructions must equal the oracle's byte for byte (no tolerance)."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

SHAPES = [(4096,), (9000,), (64, 64), (70, 130), (16, 16, 16), (20, 33, 17)]
LENGTHS = [1, 2, 15, 16, 17, 31, 32, 33, 100, 4096]


@pytest.fixture(scope="module")
def gpu():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2105_12912_gb300 import api
    return api


def _runs(shape, length, dtype=np.float32):
    """A field whose quantization codes, in storage order, come in runs of about `length`:
    a ramp along every axis whose slope changes every `length` elements (chunks restart the
    prediction, which only adds runs)."""
    n = int(np.prod(shape))
    steps = np.where((np.arange(n) // length) % 2 == 0, 1.0, 2.0).reshape(shape)
    x = np.cumsum(steps, axis=len(shape) - 1)
    return x.astype(dtype)


@pytest.mark.parametrize("select", ["rle", "rle_huff"])
@pytest.mark.parametrize("length", LENGTHS)
def test_run_expansion(gpu, orc, length, select):
    for shape in SHAPES:
        for dtype in (np.float32, np.float64):
            x = _runs(shape, length, dtype)
            ar, nb, _ = gpu.compress(torch.from_numpy(x).cuda(), 0.25, "abs", select=select)
            st, ref = orc.compress_ex(x, orc.EB_ABS, 0.25, select=gpu.SELECT[select])
            assert st == 0 and nb == ref.size and np.array_equal(ar[:nb].cpu().numpy(), ref)
            y, _ = gpu.decompress(ar, nb)
            if dtype == np.float64:
                _, yr = orc.decompress_f64(ref, x.size)
                assert np.array_equal(y.cpu().numpy().ravel().view(np.uint64), yr.view(np.uint64))
            else:
                _, yr = orc.decompress(ref, x.size)
                assert np.array_equal(y.cpu().numpy().ravel().view(np.uint32), yr.view(np.uint32))


@pytest.mark.parametrize("select", ["rle", "rle_huff", "exhaustive"])
def test_run_expansion_batch(gpu, select):
    xs = [torch.from_numpy(_runs(s, length)).cuda() for s in SHAPES for length in (1, 17, 256)]
    bc = gpu.BatchCompressor(xs, 0.25, "abs", select=select, autotune=False)
    bc.run()
    sizes, stats = bc.results()
    assert not any(stats)
    bd = gpu.BatchDecompressor([a[:n].clone() for a, n in zip(bc.archives, sizes)], [tuple(x.shape) for x in xs])
    bd.run()
    assert not any(bd.results())
    for x, a, n, y in zip(xs, bc.archives, sizes, bd.outs):
        ref, _ = gpu.decompress(a, n)
        assert torch.equal(y.view(torch.int32).ravel(), ref.view(torch.int32).ravel())
        assert float((x.double() - ref.double()).abs().max()) <= 0.25

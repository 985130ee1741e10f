"""decompress() on a stream of the caller's: everything it reads of the archive, the header
among it, is ordered behind the work already on that stream.  One buffer is refilled on a
side stream, behind a delay, with another archive of the same shape and decompressed there."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def gpu():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2105_12912_gb300 import api
    return api


@pytest.mark.parametrize("given", ["neither", "dims", "out"])
def test_refilled_buffer(gpu, given):
    shape = (130, 200)
    gen = torch.Generator().manual_seed(5)
    # (values of different ranges: the two headers differ)
    x = [torch.cumsum(torch.randn(shape, generator=gen), -1).cuda() * s for s in (1.0, 7.0)]
    ars = [gpu.compress(v, 1e-3)[:2] for v in x]
    want = gpu.decompress(ars[1][0], ars[1][1])[0].clone()
    n = max(nb for _, nb in ars)
    buf = torch.zeros(n, dtype=torch.uint8, device="cuda")
    buf[:ars[0][1]] = ars[0][0][:ars[0][1]]
    out = torch.empty(shape, device="cuda") if given == "out" else None
    side = torch.cuda.Stream()
    torch.cuda.synchronize()
    with torch.cuda.stream(side):
        torch.cuda._sleep(200_000_000)
        buf[:ars[1][1]] = ars[1][0][:ars[1][1]]
    ws = gpu.Workspace()
    y, st = gpu.decompress(buf, ars[1][1], out=out, dims=shape if given == "dims" else None, workspace=ws,
                           stream=side)
    torch.cuda.synchronize()
    assert st == 0 and torch.equal(y, want)

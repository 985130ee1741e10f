"""Launch counts of the calls against the profiler's: every kernel that ran is counted once."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def gpu():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2105_12912_gb300 import api
    return api


@pytest.mark.parametrize("kw", [{}, {"select": "rle"}, {"select": "huff"}, {"global_lorenzo": True}])
@pytest.mark.parametrize("shape", [(30000,), (300, 200), (40, 50, 60)])
def test_counts_are_the_profilers(gpu, shape, kw):
    from torch.profiler import ProfilerActivity, profile
    x = torch.cumsum(torch.randn(shape, generator=torch.Generator().manual_seed(3)), -1)
    x.view(-1)[::700] += 1e3  # outlier records
    x = x.cuda()

    b = gpu.BatchCompressor([x, x], 1e-3, plan="staged", autotune=False)

    def counted():
        ar, nb, _ = gpu.compress(x, 1e-4, **kw)
        gpu.decompress(ar, nb)
        gpu.selector_rows(x, 1e-3)
        b.run()
        torch.cuda.synchronize()

    with profile(activities=[ProfilerActivity.CUDA]):  # (the first one of a process may see nothing)
        counted()
    gpu.trace_read(reset=True)
    with profile(activities=[ProfilerActivity.CUDA]) as p:
        counted()
    got = sum(c for _, c in gpu.trace_read(reset=True).values())
    ran = sum(1 for e in p.events() if e.device_type == torch.autograd.DeviceType.CUDA and "cszp::" in e.name)
    if ran == 0:
        pytest.skip("no profiler on this machine")
    assert got == ran

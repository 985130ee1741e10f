"""GPU parity of payload placement: block counts around the 256-block groups whose totals
place the payloads, blocks of all three codecs among each other, quarters and streams that
end short, and archive buffers that end at, or before, the archive's end.

Archives must equal the oracle's byte for byte (no tolerance)."""
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


def _mixed(n, seed):
    """A walk with constant stretches, ramps of changing slope and noise, so that blocks of
    every codec occur."""
    rng = np.random.default_rng(seed)
    x = np.cumsum(rng.standard_normal(n) * 3.0)
    for s in range(0, n, 3 * 4096):
        x[s:s + 4096] = x[s]  # one run
        e = min(n, s + 2 * 4096)
        if e > s + 4096:
            k = np.arange(e - s - 4096)
            x[s + 4096:e] = x[s] + np.cumsum(np.where((k // 37) % 2, 1.0, 3.0))  # runs of 37
    return x.astype(np.float32)


@pytest.mark.parametrize("select", ["huff", "exhaustive", "rle_huff"])
@pytest.mark.parametrize("n", [1, 31, 33, 127, 129, 2049, 4095, 255 * 4096, 256 * 4096, 256 * 4096 + 1, 257 * 4096 - 5,
                               513 * 4096 + 100])
def test_payload_placement(gpu, orc, n, select):
    x = _mixed(n, n)
    ar, nb, _ = gpu.compress(torch.from_numpy(x).cuda(), 0.5, "abs", select=select)
    _, ref = orc.compress(x, orc.EB_ABS, 0.5, select=gpu.SELECT[select])
    assert nb == ref.size and np.array_equal(ar[:nb].cpu().numpy(), ref)


def test_archive_capacity(gpu):
    xd = torch.from_numpy(_mixed(300 * 4096 + 7, 3)).cuda()
    ar, nb, _ = gpu.compress(xd, 0.5, "abs")
    for cap in (nb, nb - 1, nb - 4096, nb // 2, 5000):
        buf = torch.full((nb + 64,), 0xA5, dtype=torch.uint8, device="cuda")
        _, got, st = gpu.compress(xd, 0.5, "abs", out=buf[:cap], raise_on_error=False)
        assert st == (0 if cap == nb else 5)
        assert bool((buf[cap:] == 0xA5).all())
        if st == 0:
            assert got == nb and torch.equal(buf[:nb], ar[:nb])

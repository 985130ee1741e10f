"""GPU parity of the code-book builder on histograms of extreme shape.

The builder merges many pairs at once where the histogram is dense and one pair after
another where it is sparse, so the shapes below make it take either way, switch between
them and meet ties: the archive (books, codes and streams) must be the oracle's, byte
for byte.
"""
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


def _counts(shape):
    rng = np.random.default_rng(7)
    if shape == "one":
        return [5000]
    if shape == "two":
        return [4999, 1]
    if shape == "three_ties":
        return [1, 1, 2]
    if shape == "fibonacci":  # one pair qualifies per round, the deepest tree
        f = [1, 1]
        while len(f) < 24:
            f.append(f[-1] + f[-2])
        return f
    if shape == "fibonacci_deep":  # codes of up to 32 bits: beyond both decode tables
        f = [1, 1]
        while len(f) < 33:
            f.append(f[-1] + f[-2])
        return f
    if shape == "all_ones":  # every pair qualifies
        return [1] * 1022
    if shape == "all_ones_odd":
        return [1] * 1021
    if shape == "powers":  # ties of leaves and internal nodes
        return [1 << max(0, i - 1) for i in range(17)]
    if shape == "sparse_then_dense":  # a few rare codes below a dense band
        return [1, 2, 2, 3, 5, 9, 11] + [200 + i % 7 for i in range(900)] + [40000, 90000]
    if shape == "geometric":
        return [max(1, int(200000 * 0.985 ** i)) for i in range(1000)]
    if shape == "steps":  # dense bands apart: rounds, stretches, rounds
        return [1] * 100 + [50] * 3 + [1000] * 200 + [30000] * 5 + [2, 3, 4, 7]
    return [int(v) for v in np.sort(rng.zipf(1.3, 700).clip(1, 100000))]


@pytest.mark.parametrize("shape", ["one", "two", "three_ties", "fibonacci", "fibonacci_deep", "all_ones", "all_ones_odd", "powers",
                                   "sparse_then_dense", "geometric", "steps", "zipf"])
@pytest.mark.parametrize("select", ["huff", "rle_huff"])
def test_book_shapes(gpu, orc, shape, select):
    counts = _counts(shape)
    rng = np.random.default_rng(len(counts))
    # residuals -511 .. 511 in any order; each becomes a quant code (the first of a chunk too)
    sym = rng.permutation(np.arange(-511, 512))[:len(counts)]
    delta = np.repeat(sym, counts)
    rng.shuffle(delta)
    if select == "rle_huff":
        # runs whose lengths have the same histogram shape feed the run books too
        runs = np.repeat(1 + np.arange(len(counts)), np.minimum(counts, 40))
        rng.shuffle(runs)
        runs = runs[:np.searchsorted(np.cumsum(runs), 400_000) + 1]
        vals = rng.choice(sym, runs.size)
        delta = np.concatenate([delta[:50_000], np.repeat(vals, runs)])
    x = np.concatenate([np.cumsum(c) for c in np.split(delta, np.arange(256, delta.size, 256))]).astype(np.float32)
    xd = torch.from_numpy(x).cuda()
    ar, nb, st = gpu.compress(xd, 0.5, "abs", select=select)
    _, ref = orc.compress(x, orc.EB_ABS, 0.5, select=gpu.SELECT[select])
    assert st == 0 and nb == ref.size
    assert np.array_equal(ar[:nb].cpu().numpy(), ref)
    y, _ = gpu.decompress(ar, nb)
    assert np.array_equal(y.cpu().numpy(), x)

"""The launches of an asynchronous decompression follow each other by programmatic dependent
launch.  Captured into a caller's graph and replayed they must give the call's own output,
bit for bit, for every path: fused, run and cut blocks, chunked and global prediction."""
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


@pytest.mark.parametrize("global_lorenzo", [False, True])
@pytest.mark.parametrize("shape", [(50007,), (300, 517), (40, 70, 66)])
def test_captured_decompression(gpu, shape, global_lorenzo):
    rng = np.random.default_rng(len(shape))
    x = rng.standard_normal(shape).astype(np.float32)
    for ax in range(len(shape)):
        x = np.cumsum(x, axis=ax).astype(np.float32)
    x[tuple(slice(s // 2, None) for s in shape)] = 0.0
    ar, nb, hdr = gpu.compress_with_header(torch.from_numpy(x).cuda(), 1e-3, global_lorenzo=global_lorenzo)
    ref, _ = gpu.decompress(ar, nb)
    ws = gpu.Workspace()
    out = torch.empty_like(ref)
    status = torch.full((1,), -1, dtype=torch.int32, device="cuda")
    gpu.decompress_async(ar, nb, hdr, out, status, workspace=ws)
    torch.cuda.synchronize()
    assert int(status) == 0 and torch.equal(out.view(torch.int32), ref.view(torch.int32))
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        gpu.decompress_async(ar, nb, hdr, out, status, workspace=ws)
    for _ in range(3):
        out.fill_(float("nan"))
        status.fill_(-1)
        graph.replay()
        torch.cuda.synchronize()
        assert int(status) == 0 and torch.equal(out.view(torch.int32), ref.view(torch.int32))

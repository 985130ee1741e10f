"""What follows a bounded wait that expired.  Blocks that construction gave up on hold whatever
the memory held, so nothing may be encoded from them: with the state saying so, the encoding
launches leave the archive and the context as they were, whatever the blocks hold."""
import ctypes as C
import os
import subprocess

import pytest
import torch

pytestmark = pytest.mark.gpu

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def probe(tmp_path_factory):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2105_12912_gb300 import _lib, build
    _lib.lib()
    out = str(tmp_path_factory.mktemp("probe") / "timeout_probe.so")
    subprocess.run([build.nvcc(), *build.ARCH, *build.NVFLAGS, "-shared", os.path.join(HERE, "timeout_probe.cu"),
                    build.LIB, "-o", out], check=True)
    return C.CDLL(out)


@pytest.mark.parametrize("select", ["huff", "rle", "rle_huff", "heuristic", "exhaustive"])
@pytest.mark.parametrize("shape", [(9000,), (70, 200), (20, 40, 35)])
def test_nothing_is_encoded(probe, shape, select):
    from paper_2105_12912_gb300 import api
    x = torch.cumsum(torch.randn(shape, generator=torch.Generator().manual_seed(2)), -1).cuda()
    ws = api.Workspace()
    ar, nb, _ = api.compress(x, 1e-3, select=select, workspace=ws)
    keep = ar[:nb].clone()
    out = torch.full_like(ar, 0xa5)
    for spoil in (0, 1):
        assert probe.probe_encode(C.c_void_p(x.data_ptr()), len(shape), (C.c_uint64 * 3)(*shape), api.SELECT[select],
                                  C.c_void_p(ws.buf.data_ptr()), C.c_void_p(out.data_ptr()), C.c_uint64(out.numel()),
                                  spoil) == 0
        assert bool((out == 0xa5).all())
    ar, nb, _ = api.compress(x, 1e-3, select=select, workspace=ws)
    assert torch.equal(ar[:nb], keep)


@pytest.mark.parametrize("global_lorenzo", [False, True])
@pytest.mark.parametrize("shape", [(9000,), (70, 200), (20, 40, 35)])
def test_nothing_is_decoded(probe, shape, global_lorenzo):
    """The same after an expired wait in decompression's set-up: the output stays as it was."""
    from paper_2105_12912_gb300 import api
    x = torch.cumsum(torch.randn(shape, generator=torch.Generator().manual_seed(4)), -1)
    x[: shape[0] // 3] = 0.0
    x = x.cuda()
    ws = api.Workspace()
    ar, nb, hdr = api.compress_with_header(x, 1e-3, radius=32, workspace=ws, global_lorenzo=global_lorenzo)
    out = torch.full_like(x, -7.0)
    assert probe.probe_decode(C.c_void_p(ar.data_ptr()), C.c_uint64(nb), hdr, len(shape), (C.c_uint64 * 3)(*shape),
                              C.c_void_p(ws.buf.data_ptr()), C.c_void_p(out.data_ptr())) == 0
    assert bool((out == -7.0).all())
    y, st = api.decompress(ar, nb, workspace=ws)
    assert st == 0 and float((x.double() - y.double()).abs().max()) <= api.header(ar)["eb_f"]

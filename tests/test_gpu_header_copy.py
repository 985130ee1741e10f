"""csz_archive_head / csz_decompress_with_header and the header that comes back with a
compression: the same output as csz_decompress, and its refusals -- a copy that is not the
archive's, the other element type, a buffer too short for a header."""
import ctypes as C

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


def _ptr(t):
    return C.c_void_p(t.data_ptr())


@pytest.mark.parametrize("dtype", [torch.float32, torch.float64])
@pytest.mark.parametrize("shape", [(10007,), (70, 131), (19, 23, 37)])
def test_header_copy(gpu, shape, dtype):
    from paper_2105_12912_gb300 import _lib
    lib = _lib.lib()
    x = torch.cumsum(torch.randn(shape, generator=torch.Generator().manual_seed(1)), -1).to(dtype).cuda()
    ar, nb, _ = gpu.compress(x, 1e-3)
    f64 = int(dtype == torch.float64)
    hdr, nd, esz, dims = (C.c_uint8 * 128)(), C.c_int(), C.c_int(), (C.c_uint64 * 3)()
    assert lib.csz_archive_head(_ptr(ar), nb, hdr, C.byref(nd), dims, C.byref(esz), None) == 0
    assert bytes(hdr) == bytes(ar[:128].cpu().numpy()) and tuple(dims[:nd.value]) == shape and esz.value == (8 if f64 else 4)
    assert lib.csz_archive_head(_ptr(ar), 127, hdr, C.byref(nd), dims, C.byref(esz), None) == 4
    if not f64:
        ar2, nb2, h2 = gpu.compress_with_header(x, 1e-3)
        assert nb2 == nb and h2 == bytes(hdr)
    ref = torch.empty_like(x)
    ws = torch.empty(gpu.workspace_bytes(shape), dtype=torch.uint8, device="cuda")
    fn = lib.csz_decompress_f64 if f64 else lib.csz_decompress
    assert fn(_ptr(ar), nb, _ptr(ref), ref.numel(), _ptr(ws), ws.numel(), None) == 0
    out = torch.full_like(x, float("nan"))

    def call(h, wide=f64, n=nb):
        return lib.csz_decompress_with_header(_ptr(ar), n, h, wide, _ptr(out), out.numel(), _ptr(ws), ws.numel(), None)

    assert call(hdr) == 0 and torch.equal(out, ref)
    py, _ = gpu.decompress(ar, nb)
    assert py.dtype == dtype and torch.equal(py, ref)
    assert call(hdr, wide=1 - f64) == 1
    assert call(hdr, n=100) == 4
    other = (C.c_uint8 * 128).from_buffer_copy(bytes(hdr))
    other[32] ^= 1  # the user's bound: informational, but not the archive's own
    assert call(other) == 4
    other = (C.c_uint8 * 128).from_buffer_copy(bytes(hdr))
    other[0] ^= 1
    assert call(other) == 4

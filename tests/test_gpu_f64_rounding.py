"""GPU parity of double fields where the prequantization's integer path hands over to the
exact decision: values at every distance from the half points, zeros of both signs,
subnormals, and bounds whose quantization step lies outside the integer path's exponents.
Shapes: a TMA-described 3-D field, and ragged ones whose rows TMA cannot describe.

Codes, archives and reconstructions must equal the oracle's byte for byte, so there is no
tolerance."""
import numpy as np
import pytest
import torch

from test_gpu_f64 import _parity

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def gpu():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2105_12912_gb300 import api
    return api


@pytest.mark.parametrize("eb", [0.37, 2.0 ** -30, 1e250, 1e-250, 1e281, 1e-281])
@pytest.mark.parametrize("shape", [(32, 32, 48), (17, 18, 35), (37, 131), (4101,)])
def test_f64_around_half_points(gpu, orc, eb, shape):
    st, eb_d, step, rstep = orc.eb_params_f64(orc.EB_ABS, eb)
    vals = [0.0, -0.0, 5e-324, -2.2e-308]
    for k in [0, 1, 2, 77, 4096, 99991, 2 ** 20 + 7, 2 ** 24 + 1, 2 ** 26 - 5]:
        for j in range(1, 46):
            for d in (2.0 ** -j, -(2.0 ** -j)):
                v = (k + 0.5 + d) * step
                vals += [v, -v]
    n = int(np.prod(shape))
    x = np.resize(np.array(vals), n).reshape(shape)
    assert _parity(gpu, orc, x, eb, mode="abs") == 0

"""decompress() of what holds no whole header: corrupt, whether or not it has an address."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [0, 1, 127])
def test_no_whole_header(n):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2105_12912_gb300 import _lib, api
    with pytest.raises(_lib.CszError) as e:
        api.decompress(torch.zeros(n, dtype=torch.uint8, device="cuda"))
    assert e.value.status == 4  # CSZ_E_CORRUPT

"""The FFT passes of the large mesh sizes, as test_fft_sizes_gpu.py has the others."""
import pytest

from test_fft_sizes_gpu import solve_error
from test_parity_gpu import pm  # noqa: F401  (a fixture)

pytestmark = pytest.mark.gpu


def room(n, word):
    """Skips where the context (33 fields and the spectra's extra plane) and the check's FP64 arrays do not fit."""
    import torch
    torch.cuda.empty_cache()
    need = n ** 3 * (36 * word + 12 * 8)
    if torch.cuda.mem_get_info()[0] < need:
        pytest.skip("needs %d GB of device memory" % (need >> 30))


@pytest.mark.parametrize("n", [96, 192, 256, 384, 512, 576, 768, 1024])
def test_mixed_large_sizes(pm, n):  # noqa: F811
    """FP32 transforms: about sqrt(log2 N^3) roundings of 2^-24 each way, below 5e-7."""
    room(n, 4)
    assert solve_error(pm, n, pm.PM_MIXED) < 5e-7


@pytest.mark.parametrize("n", [48, 192, 256, 384, 432, 512, 576, 648, 768])
def test_fp64_large_sizes(pm, n):  # noqa: F811
    room(n, 8)
    assert solve_error(pm, n, pm.PM_FP64) < 1e-14

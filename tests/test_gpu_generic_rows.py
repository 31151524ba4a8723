"""GPU: SMSM_FLAG_GENERIC_KERNELS reaches the shape-generic row transforms, and both forms agree.

The two-register-DFT transforms (csrc/rowfft.cu) and the Stockham passes (csrc/operators.cu) round differently, so equal
bits at every length would mean that the flag reaches one of them only.  Tolerance: each is within the FP32 operator
bar of test_gpu_parity.py (1e-5) of the same result.
"""
import pytest
import torch

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.fixture(scope="module")
def smsm():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1901_01893_gb300 import _build, smsm as mod

    _build.build()
    mod.lib()
    return mod


def test_generic_row_transforms(smsm):
    differ = 0
    for N in (48, 64, 72, 96, 108, 128, 144, 192, 256):
        x = torch.randn(3, N, N, dtype=torch.complex64, device=DEV)
        for inverse in (False, True):
            a, b = (smsm.Plan(1, 1, 2, N, 2, flags=f).fft2c(x, inverse=inverse)
                    for f in (0, smsm.SMSM_FLAG_GENERIC_KERNELS))
            assert (torch.linalg.vector_norm(a - b) / torch.linalg.vector_norm(a)).item() < 2e-5
            differ += not torch.equal(a, b)
    assert differ > 0

"""GPU: the tensor-core Gram's complex128 result where the sum of its FP32 partials leaves FP32's range.

k-space of 4e17: a Gram entry is some 2e35 times the number of patches, above 3.4e38 in total and below it in every
partial.  Tolerance: the FP32 operator bar of test_gpu_parity.py, 1e-5.
"""
import numpy as np
import pytest
import torch

import oracle as O

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


@pytest.mark.parametrize("Ns,r,N", [(2, 3, 64), (4, 6, 128)])
def test_gram_beyond_fp32_range(smsm, Ns, r, N):
    rng = np.random.default_rng(N)
    u = (1 + 0.2 * (rng.standard_normal((1, Ns, N, N)) + 1j * rng.standard_normal((1, Ns, N, N)))).astype(np.complex64)
    s = np.float32(4.5e17 if N == 64 else 2.2e17)
    ref = O.gram((u * s).astype(np.complex128), r)
    assert np.abs(ref).max() > 3.4028e38
    G = smsm.Plan(1, Ns, 2, N, r).hankel_gram(torch.from_numpy(u * s).to(DEV)).cpu().numpy()
    assert O.nrmse(G / 1e38, ref / 1e38) < 1e-5

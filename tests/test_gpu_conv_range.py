"""GPU: the convolution's split of an activation (csrc/cnn.cu) where BF16 rounds it to infinity.

One pixel of the input is infinite, or finite and above the largest BF16 value.  Against the same two layers in plain
float64 torch (a complex product as its four real ones, CReLU as max(v, 0)) with weights that are BF16 values: the same
NaNs and infinities, and 1e-5 on what is finite (the forward bar of test_gpu_cnn.py).
"""
import numpy as np
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


def conv64(h, w):
    """h [1][2][H][W] (re, im), w [9] complex -> the same of the complex 3 x 3 cross-correlation, zero padding"""
    p = torch.nn.functional.pad(h, (1, 1, 1, 1))
    H, W = h.shape[2:]
    re = im = 0
    for k in range(9):
        a, b = p[:, 0, k // 3:k // 3 + H, k % 3:k % 3 + W], p[:, 1, k // 3:k // 3 + H, k % 3:k % 3 + W]
        re, im = re + w[k].real * a - w[k].imag * b, im + w[k].real * b + w[k].imag * a
    return torch.stack([re, im], 1)


@pytest.mark.parametrize("value", [np.inf, -np.inf, np.nan, 3.4e38, -3.4e38, 3.397e38, 3.385e38])
@pytest.mark.parametrize("sign", [1, -1])
def test_large_and_infinite_activations(smsm, value, sign):
    H, W = 12, 70
    rng = np.random.default_rng(5)
    scale = 2.0 ** -12 if np.isfinite(value) else 1.0
    w = [(rng.integers(4, 9, 9) + sign * 1j * rng.integers(4, 9, 9)) / 8 * s for s in (scale, 1.0)]
    a = (rng.standard_normal((1, 1, H, W)) + 1j * rng.standard_normal((1, 1, H, W))).astype(np.complex64)
    a[0, 0, 5, 33] = np.complex64(complex(np.float32(value), 0.5))
    net = smsm.CNN(1, H, W, width=1, layers=2, max_batch=1)
    net.set_params(torch.from_numpy(np.concatenate([w[0], [0], w[1], [0]]).astype(np.complex64)).to(DEV))
    out = net.forward(torch.from_numpy(a).to(DEV)).cpu()
    x = torch.from_numpy(np.stack([a[:, 0].real, a[:, 0].imag], 1).astype(np.float64))
    h = conv64(x, w[0])
    ref = x + conv64(torch.where(h > 0, h, torch.zeros_like(h)), w[1])  # (a NaN is not above 0: CReLU gives 0)
    ref = torch.where(ref.abs() > 3.4028e38, torch.sign(ref) * np.inf, ref)  # FP32's range
    got = torch.stack([out[:, 0].real, out[:, 0].imag], 1).double()
    assert torch.equal(got.isnan(), ref.isnan())
    assert torch.equal(torch.where(got.isinf(), got, 0), torch.where(ref.isinf(), ref, 0))
    far = torch.zeros_like(ref, dtype=torch.bool)
    far[:, :, 3:8, 31:36] = True  # the pixels that see the large one; elsewhere values are of order one
    for part in (far, ~far):
        m = part & ref.isfinite()
        if m.any():
            assert ((got - ref)[m].norm() / ref[m].norm()).item() < 1e-5

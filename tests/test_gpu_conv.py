"""GPU parity of the tensor-core convolution (csrc/cnn.cu) at the edges of its tiles.

Image widths around the 64-column strips, images smaller than a tile, channel counts that are no multiple of the 8
staged at a time, more than 64 output channels (several column blocks), non-square images.  Two layers, so that
the first and the CReLU form are both met.  Tolerance: the forward bar of test_gpu_cnn.py, 1e-5 per sample.
"""
import numpy as np
import pytest
import torch

import oracle as O
from oracle import cnn as OC

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


@pytest.mark.parametrize("B,width,H,W,n", [
    (1, 1, 5, 3, 2), (9, 65, 7, 64, 1), (4, 130, 6, 65, 1), (70, 20, 9, 66, 1), (16, 17, 33, 128, 2), (2, 8, 1, 129, 1),
])
def test_conv_tile_edges(smsm, B, width, H, W, n):
    rng = np.random.default_rng(B + width)
    cr = lambda *s: rng.standard_normal(s) + 1j * rng.standard_normal(s)  # noqa: E731
    shapes = OC.layer_shapes(B, width, 2)
    flat = np.concatenate([np.concatenate([cr(co * ci * 9) / np.sqrt(9 * ci), 0.1 * cr(co)]) for co, ci in shapes])
    t = torch.view_as_real(torch.from_numpy(flat.astype(np.complex64)))
    v = torch.view_as_complex(t.to(torch.bfloat16).double().contiguous()).numpy()  # the weights the kernels use
    params, at = [], 0
    for co, ci in shapes:
        k = co * ci * 9
        params.append((v[at:at + k].reshape(co, ci, 3, 3), v[at + k:at + k + co]))
        at += k + co
    a = cr(n, B, H, W).astype(np.complex64)
    net = smsm.CNN(B, H, W, width=width, layers=2, max_batch=n)
    net.set_params(torch.from_numpy(flat.astype(np.complex64)).to(DEV))
    out = net.forward(torch.from_numpy(a).to(DEV)).cpu().numpy()
    for s in range(n):
        assert O.nrmse(out[s], OC.forward(a[s].astype(np.complex128), params)) < 1e-5

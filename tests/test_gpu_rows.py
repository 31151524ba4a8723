"""GPU parity at the edges of the two-register-DFT row transforms (csrc/rowfft.cu), of the column stages' two-step
transforms (csrc/colalias.cu, csrc/colfast.cu) and of the tensor-core Gram's partial layout (csrc/gram_tc.cu).

Transforms: every length with a kernel of its own and lengths next to them that keep the older kernels, through
fft2c.  Normal operator: shot counts on both sides of the rule (4), integer and sub-pixel CAIPI shifts, through a
short solve.  Gram: 2C at and just past the tile edges, ragged patch rows.  Tolerances: the bars of
test_gpu_parity.py, 1e-5 for an FP32 operator and 2e-5 per slice for a solve.
"""
import numpy as np
import pytest
import torch

import oracle as O
from paper_1901_01893_gb300 import synth

pytestmark = pytest.mark.gpu

OP_TOL = 1e-5
SOLVE_TOL = 2e-5
DEV = "cuda:0"


@pytest.fixture(scope="module")
def smsm():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1901_01893_gb300 import _build, smsm as mod

    _build.build()
    mod.lib()
    return mod


def c64(a):
    return torch.from_numpy(np.ascontiguousarray(a).astype(np.complex64)).to(DEV)


def crandn(seed, *s):
    rng = np.random.default_rng(seed)
    return (rng.standard_normal(s) + 1j * rng.standard_normal(s)).astype(np.complex64)


@pytest.mark.parametrize("N", [32, 36, 48, 64, 72, 96, 108, 128, 144, 162, 192, 256, 324])
def test_transform_lengths(smsm, N):
    p = smsm.Plan(1, 1, 2, N, 2)
    img = crandn(N, 3, N, N)
    k = p.fft2c(c64(img)).cpu().numpy()
    assert O.nrmse(k, O.fft2c(img.astype(np.complex128))) < OP_TOL
    assert O.nrmse(p.fft2c(c64(k), inverse=True).cpu().numpy(), img) < OP_TOL


@pytest.mark.parametrize("L,Ns,N,div", [
    (2, 4, 48, 2), (2, 3, 72, 2), (2, 2, 64, 2), (1, 1, 96, 1), (2, 4, 128, 4), (2, 6, 72, 2), (2, 3, 108, 3),
    (3, 2, 64, 3), (2, 4, 64, 3), (2, 6, 48, 2), (2, 8, 64, 2), (3, 4, 128, 3), (2, 2, 96, 2),
])
def test_normal_operator_lengths(smsm, L, Ns, N, div):
    g = synth.make_group(L, Ns, 6, N, 5)
    _, y = O.make_data(g, 30.0, div)
    y = y / np.sqrt(np.mean(np.abs(y) ** 2))
    K, J, lam = 2, 3, 1e-2
    ref = O.reconstruct(y, g["sens"], 2, dict(K=K, J=J, lam=lam), Ldiv=div)
    p = smsm.Plan(L, Ns, 6, N, 2, caipi_div=div)
    p.set_sens(c64(g["sens"]))
    x, rep = p.reconstruct(c64(y), params=smsm.default_params(lam=lam, outer_iters=K, cg_iters=J))
    assert rep.status == 0
    assert float(np.max(O.nrmse(x.cpu().numpy(), ref, axis=(1, 2, 3)))) < SOLVE_TOL


@pytest.mark.parametrize("Ns,r,N", [
    (1, 4, 24), (2, 3, 32), (4, 4, 48), (1, 9, 32), (3, 5, 36), (8, 4, 32), (2, 8, 48), (4, 6, 36), (1, 1, 18),
])
def test_gram_tile_edges(smsm, Ns, r, N):
    p = smsm.Plan(2, Ns, 2, N, r)
    x = crandn(Ns * r, 2, Ns, N, N)
    G = p.hankel_gram(c64(x)).cpu().numpy()
    assert p.device_status() == 0
    assert O.nrmse(G, O.gram(x.astype(np.complex128), r)) < OP_TOL
    assert np.array_equal(G, np.conj(np.swapaxes(G, 1, 2)))

"""GPU parity of the column stage of A and A^H over the lengths of its kernels (csrc/colwarp.cu).

Every M = N/Ns with a kernel of its own, odd coil counts (a last set of coils that is not full, fewer coils than
a set), shot counts on both sides of a kernel's limit and the geometries that fall back to k_col; with and without
the shot phase, batch of two.  Tolerance: the FP32 operator bar of test_gpu_parity.py, 1e-5.
"""
import numpy as np
import pytest
import torch

import oracle as O

pytestmark = pytest.mark.gpu

OP_TOL = 1e-5
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


@pytest.mark.parametrize("L,Ns,Nc,N,Ldiv", [
    (1, 8, 3, 64, 2), (3, 6, 7, 48, 3), (2, 6, 5, 72, 2), (1, 4, 1, 48, 4), (2, 8, 9, 128, 3), (1, 4, 5, 72, 1),
    (2, 6, 3, 108, 2), (1, 3, 12, 72, 3), (2, 8, 5, 192, 2), (2, 3, 9, 96, 4), (1, 2, 3, 64, 1), (2, 3, 4, 108, 2),
    (1, 1, 2, 48, 1), (2, 3, 3, 144, 2), (2, 2, 3, 108, 3), (3, 4, 6, 256, 3), (1, 2, 5, 144, 2), (2, 2, 3, 192, 2),
    (1, 1, 3, 108, 2), (3, 2, 3, 256, 3), (1, 1, 2, 144, 1), (2, 1, 3, 192, 2), (3, 1, 2, 256, 3), (2, 4, 2, 512, 2),
    (3, 8, 2, 64, 3), (3, 6, 4, 96, 2),
])
@pytest.mark.parametrize("phase", [False, True])
def test_forward_adjoint_lengths(smsm, L, Ns, Nc, N, Ldiv, phase):
    rng = np.random.default_rng(N + 10 * Ns + Nc)
    cr = lambda *s: rng.standard_normal(s) + 1j * rng.standard_normal(s)  # noqa: E731
    S, D = cr(L, Nc, N, N) / np.sqrt(Nc), 2
    x, y = cr(D, L, 1 if phase else Ns, N, N), cr(D, Ns, Nc, N // Ns, N)
    ph = np.exp(1j * rng.uniform(-np.pi, np.pi, (D, L, Ns, N, N))) if phase else None
    p = smsm.Plan(L, Ns, Nc, N, 2, caipi_div=Ldiv, batch=D)
    p.set_sens(c64(S))
    kw = dict(phase=c64(ph)) if phase else {}
    yg, xg = p.forward(c64(x), **kw).cpu().numpy(), p.adjoint(c64(y), **kw).cpu().numpy()
    assert p.device_status() == 0
    for d in range(D):
        kd = dict(phase=ph[d]) if phase else {}
        assert O.nrmse(yg[d], O.forward(x[d], S, Ldiv=Ldiv, **kd)) < OP_TOL
        assert O.nrmse(xg[d], O.adjoint(y[d], S, L, Ldiv=Ldiv, **kd)) < OP_TOL

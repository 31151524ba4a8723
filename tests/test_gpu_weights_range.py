"""GPU: the IRLS weights (csrc/invsqrt.cu) over what a solve may meet: an empty slice, data of any scale.

Tolerance: the FP32 whole-solve bar of test_gpu_parity.py, 2e-5 per slice, against the FP64 oracle.  The problem
scales with its data when lambda does (W has the inverse scale), so one oracle solve serves every scale.
"""
import numpy as np
import pytest
import torch

import oracle as O
from paper_1901_01893_gb300 import synth

pytestmark = pytest.mark.gpu

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


@pytest.mark.parametrize("Ns,r,N", [(4, 5, 64), (1, 4, 32), (8, 6, 48)])
def test_an_empty_slice_leaves_the_others_alone(smsm, Ns, r, N):
    # coil maps that are zero over a whole slice (all air): its Gram is exactly zero
    g = synth.make_group(2, Ns, 6, N, 11)
    S = g["sens"].copy()
    S[1] = 0
    _, y = O.make_data(dict(g, sens=S), 30.0)
    y = y / np.sqrt(np.mean(np.abs(y) ** 2))
    K, J, lam = 3, 3, 1e-2
    rp = {}
    ref = O.reconstruct(y, S, r, dict(K=K, J=J, lam=lam), report=rp)
    p = smsm.Plan(2, Ns, 6, N, r)
    p.set_sens(c64(S))
    x, rep = p.reconstruct(c64(y), params=smsm.default_params(lam=lam, outer_iters=K, cg_iters=J))
    x = x.cpu().numpy()
    assert rep.status == 0
    assert O.nrmse(x[0], ref[0]) < SOLVE_TOL
    assert np.all(x[1] == 0)
    assert rep.eps[0] == pytest.approx(rp["hist"][0]["eps"], rel=1e-5)


@pytest.mark.parametrize("e", [-50, -45, -30, 0, 20, 30, 45, 55])
def test_data_of_any_scale(smsm, e):
    g = synth.make_group(2, 4, 6, 48, 12)
    _, y = O.make_data(g, 30.0)
    y = y / np.sqrt(np.mean(np.abs(y) ** 2))
    K, J, lam, s = 3, 3, 1e-2, 2.0 ** e
    rp = {}
    ref = O.reconstruct(y, g["sens"], 5, dict(K=K, J=J, lam=lam), report=rp)
    p = smsm.Plan(2, 4, 6, 48, 5)
    p.set_sens(c64(g["sens"]))
    x, rep = p.reconstruct(c64(y * s), params=smsm.default_params(lam=lam * s, outer_iters=K, cg_iters=J))
    assert rep.status == 0 and list(rep.sweeps)[:K] == [0] * K
    assert float(np.max(O.nrmse(x.cpu().numpy().astype(complex) / s, ref, axis=(1, 2, 3)))) < SOLVE_TOL
    assert rep.eps[0] / s ** 2 == pytest.approx(rp["hist"][0]["eps"], rel=1e-5)


@pytest.mark.parametrize("eps0", [1e-5, 1.2e-5, 2e-5, 1e-4])
def test_an_indefinite_gram_takes_the_eigensolver(smsm, eps0):
    # BF16 split Gram of shots that are constants 1.0078125 +- 0.0038 over k-space: the part each value loses to the
    # first BF16 piece alternates in sign over the shots, so it is coherent and orthogonal to the data; three products
    # leave out its square, -1.4e-5 of the largest eigenvalue: more than eps, or a part of it.  The eigensolver clamps it.
    # The bar: no further from the oracle than the solve that uses the eigensolver throughout (its own error there is
    # rounding next to eps), with the short solve's bar on top.
    v = 1.0078125 + 0.0038 * np.array([1, -1] * 4)
    x0 = np.ones((1, 8, 64, 64)) * v[None, :, None, None] * (1 + 0j)
    g = synth.make_group(1, 8, 4, 64, 3)
    _, y = O.make_data(g, 30.0)
    y = y / np.sqrt(np.mean(np.abs(y) ** 2))
    par = dict(eps0_rel=eps0, eps_min_rel=1.0)
    ref = O.reconstruct(y, g["sens"], 2, dict(K=1, J=2, lam=1e-1, **par), x0=x0)
    p = smsm.Plan(1, 8, 4, 64, 2, precision=smsm.SMSM_PRECISION_BF16_SPLIT)
    p.set_sens(c64(g["sens"]))
    err = {}
    for cold in (0, 1):
        prm = smsm.default_params(lam=1e-1, outer_iters=1, cg_iters=2, warm=1, eig_cold=cold, **par)
        x, rep = p.reconstruct(c64(y), x=c64(x0), params=prm)
        assert rep.status == 0
        err[cold] = float(np.max(O.nrmse(x.cpu().numpy(), ref, axis=(1, 2, 3))))
    print("errors", err)
    assert err[0] < 2 * err[1] + SOLVE_TOL


@pytest.mark.parametrize("Ns,r,N", [(4, 4, 32), (4, 6, 48), (8, 6, 48)])
def test_matrices_left_to_the_eigensolver_start_warm(smsm, Ns, r, N):
    # a start 1e-3 of the data's size: from the second outer iteration on c/eps is beyond the quadrature's range, and
    # from the third on the eigensolver has the eigenvectors of the iteration before.  Fewer sweeps than from scratch
    # in every one of them, and no further from the oracle (the bar of the test next to this in test_gpu_weights.py).
    g = synth.make_group(2, Ns, 6, N, 4)
    _, y = O.make_data(g, 30.0)
    y = y / np.sqrt(np.mean(np.abs(y) ** 2))
    x0 = O.adjoint(y, g["sens"], 2) * 1e-3
    K, J, lam = 6, 3, 1e-3
    ref = O.reconstruct(y, g["sens"], r, dict(K=K, J=J, lam=lam), x0=x0)
    p = smsm.Plan(2, Ns, 6, N, r)
    p.set_sens(c64(g["sens"]))
    err, sweeps = {}, {}
    for cold in (0, 1):
        prm = smsm.default_params(lam=lam, outer_iters=K, cg_iters=J, warm=1, eig_cold=cold)
        x, rep = p.reconstruct(c64(y), x=c64(x0), params=prm)
        assert rep.status == 0
        err[cold], sweeps[cold] = float(np.max(O.nrmse(x.cpu().numpy(), ref, axis=(1, 2, 3)))), list(rep.sweeps)[:K]
    print("errors", err, "sweeps", sweeps)
    assert sweeps[0][0] == 0 and sweeps[0][1] > 0
    assert all(a < b for a, b in zip(sweeps[0][2:], sweeps[1][2:]))
    assert err[0] < 2 * err[1] + SOLVE_TOL

"""GPU: batches beyond the scratch of the Gram and weight steps, and the warm-started eigensolvers of IRLS weights.

Scratch: more matrices than one launch takes (65 at C = 144, 17 at C = 288), in one lane (several launches) and in
four (each lane its own part).  The lanes give the same bits, and every direction is within the FP32 whole-solve bar
of test_gpu_parity.py (2e-5 per slice) of the same direction in a plan that needs one launch.

Warm start: asked for by a rotation threshold, the eigensolvers make every weight; from the second outer iteration
on they start from the eigenvectors before, with fewer sweeps than from scratch and within the same bar of the oracle.
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


@pytest.mark.parametrize("Ns,r,N,D", [(4, 6, 24, 70), (8, 6, 48, 20)])
def test_batches_beyond_the_scratch(smsm, Ns, r, N, D):
    S = synth.make_group(1, Ns, 6, N, 1)["sens"]
    ys = []
    for d in range(D):
        _, y = O.make_data(dict(synth.make_group(1, Ns, 6, N, 100 + d), sens=S), 30.0)
        ys.append(y / np.sqrt(np.mean(np.abs(y) ** 2)))
    y = c64(np.stack(ys))
    prm = dict(lam=1e-2, outer_iters=2, cg_iters=3)
    p = smsm.Plan(1, Ns, 6, N, r, batch=D)
    p.set_sens(c64(S))
    x = {}
    for lanes in (1, 4):
        xl, rep = p.reconstruct(y, params=smsm.default_params(lanes=lanes, **prm))
        assert rep.status == 0 and rep.lanes == lanes
        x[lanes] = xl.cpu().numpy()
    assert np.array_equal(x[1], x[4])
    few = smsm.Plan(1, Ns, 6, N, r, batch=10)
    few.set_sens(c64(S))
    for d0 in range(0, D, 10):
        ref = few.reconstruct(y[d0:d0 + 10].contiguous(), params=smsm.default_params(**prm))[0].cpu().numpy()
        assert float(np.max(O.nrmse(x[1][d0:d0 + 10], ref, axis=(2, 3, 4)))) < SOLVE_TOL


@pytest.mark.parametrize("Ns,r,N,tol", [(4, 5, 48, 1e-6), (8, 6, 48, 2e-6)])
def test_eigensolvers_start_warm_for_irls_weights(smsm, Ns, r, N, tol):
    g = synth.make_group(2, Ns, 6, N, 21)
    _, y = O.make_data(g, 30.0)
    y = y / np.sqrt(np.mean(np.abs(y) ** 2))
    K, J, lam = 4, 3, 1e-2
    ref = O.reconstruct(y, g["sens"], r, dict(K=K, J=J, lam=lam))
    p = smsm.Plan(2, Ns, 6, N, r)
    p.set_sens(c64(g["sens"]))
    sweeps = {}
    for cold in (0, 1):
        prm = smsm.default_params(lam=lam, outer_iters=K, cg_iters=J, eig_tol=tol, eig_cold=cold)
        x, rep = p.reconstruct(c64(y), params=prm)
        assert rep.status == 0
        assert float(np.max(O.nrmse(x.cpu().numpy(), ref, axis=(1, 2, 3)))) < SOLVE_TOL
        sweeps[cold] = list(rep.sweeps)[:K]
    print("sweeps", sweeps)
    assert min(sweeps[0]) > 0 and all(a < b for a, b in zip(sweeps[0][1:], sweeps[1][1:]))

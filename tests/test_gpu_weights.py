"""GPU parity of the solve's FP32 Gram (csrc/gram_lag.cu) and of the IRLS weights formed without an
eigen-decomposition (csrc/invsqrt.cu).

Neither is an output, so they are tested through a short solve against the FP64
oracle, at the edges of the kernels' tiles: one 16 x 16 block, a ragged last block, the most blocks of one
CTA (C = 192), the first and last sizes of the four-CTA form (C = 196, 294).  Tolerance: the FP32
whole-solve bar of test_gpu_parity.py (2e-5 per slice), which the eigensolver's weights are held to.
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


def problem(L, Ns, Nc, N, seed):
    g = synth.make_group(L, Ns, Nc, N, seed)
    xt, y = O.make_data(g, 30.0)
    return g, y / np.sqrt(np.mean(np.abs(y) ** 2))


def worst(x, ref):
    return float(np.max(O.nrmse(x, ref, axis=(1, 2, 3))))


@pytest.mark.parametrize("L,Ns,N,r", [
    (1, 1, 32, 4),    # C = 16: one block
    (2, 2, 32, 3),    # C = 18: ragged second block
    (1, 3, 48, 8),    # C = 192: 78 blocks on one CTA
    (1, 4, 32, 7),    # C = 196: 91 blocks on four CTAs, ragged
    (1, 6, 48, 7),    # C = 294: 190 blocks on four CTAs
    (1, 1, 16, 8),    # Gram: half a row tile, a core of two rows and columns
    (2, 2, 36, 2),    # Gram: ragged second row tile, 3 lags
    (1, 1, 24, 12),   # Gram: 23 lags, one shot per task
    (1, 2, 48, 10),   # Gram: 19 lags, one shot per task, two shots
    (3, 3, 96, 1),    # Gram: no edges, odd shot count
])
def test_solve_parity_at_block_edges(smsm, L, Ns, N, r):
    g, y = problem(L, Ns, 6, N, 3)
    K, J, lam = 3, 3, 1e-2
    ref = O.reconstruct(y, g["sens"], r, dict(K=K, J=J, lam=lam))
    p = smsm.Plan(L, Ns, 6, N, r)
    p.set_sens(c64(g["sens"]))
    x, rep = p.reconstruct(c64(y), params=smsm.default_params(lam=lam, outer_iters=K, cg_iters=J))
    e = worst(x.cpu().numpy(), ref)
    print(f"C = {Ns * r * r}: {e:.2e}")
    assert rep.status == 0 and list(rep.sweeps)[:K] == [0] * K  # no eigen-decomposition was made
    assert e < SOLVE_TOL


def test_start_far_below_the_iterates_takes_the_eigensolver(smsm):
    # a warm start 1e-3 of the data's size: eps_1 comes from its Gram, 1e-6 of the later ones, so
    # from the second outer iteration on the weights are the eigensolver's.  Its own error there
    # (FP32 noise next to eps) is the bar: no further from the oracle than the solve that uses
    # the eigensolver throughout, with the short solve's bar on top.
    L, Ns, Nc, N, r = 2, 4, 6, 32, 4
    g, y = problem(L, Ns, Nc, N, 4)
    x0 = O.adjoint(y, g["sens"], L) * 1e-3
    ref = O.reconstruct(y, g["sens"], r, dict(K=2, J=3, lam=1e-3), x0=x0)
    err = {}
    for cold in (0, 1):
        p = smsm.Plan(L, Ns, Nc, N, r)
        p.set_sens(c64(g["sens"]))
        prm = smsm.default_params(lam=1e-3, outer_iters=2, cg_iters=3, warm=1, eig_cold=cold)
        x, rep = p.reconstruct(c64(y), x=c64(x0), params=prm)
        assert rep.status == 0
        assert rep.sweeps[1] > 0 and (rep.sweeps[0] > 0) == bool(cold)
        err[cold] = worst(x.cpu().numpy(), ref)
    print("errors", err)
    assert err[0] < 2 * err[1] + SOLVE_TOL

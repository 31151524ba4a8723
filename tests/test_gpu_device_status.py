"""GPU: a bounded wait that ran out is heard by the caller.

No wait can be made to run out here (the copies and matrix products they wait for always end), so the device flag
is raised from the host, as the kernel would.
"""
import ctypes

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
    lib = mod.lib()
    for f in (lib.smsm_cnn_raise_for_test, lib.smsm_plan_raise_for_test):
        f.argtypes, f.restype = [ctypes.c_void_p, ctypes.c_int], ctypes.c_int
    return mod


def test_network_reports_and_clears_its_flag(smsm):
    net = smsm.CNN(2, 16, 16, width=4, layers=2, max_batch=1)
    net.set_params(torch.randn(net.count, dtype=torch.complex64, device=DEV))
    a = torch.randn(1, 2, 16, 16, dtype=torch.complex64, device=DEV)
    net.forward(a)
    assert net.device_status() == 0
    smsm.lib().smsm_cnn_raise_for_test(net._h, smsm.SMSM_ERR_TIMEOUT)
    net.forward(a)  # asynchronous: no error yet
    assert net.device_status() == smsm.SMSM_ERR_TIMEOUT
    assert net.device_status() == 0  # once
    smsm.lib().smsm_cnn_raise_for_test(net._h, smsm.SMSM_ERR_TIMEOUT)
    with pytest.raises(smsm.SmsmError) as e:
        net.gradients(a, a)
    assert e.value.status == smsm.SMSM_ERR_TIMEOUT
    loss, _ = net.gradients(a, a)
    assert loss > 0


def test_reports_carry_the_plans_flag(smsm):
    p = smsm.Plan(1, 2, 2, 32, 2)
    p.set_sens(torch.randn(1, 2, 32, 32, dtype=torch.complex64, device=DEV))
    y = torch.randn(p.y_shape, dtype=torch.complex64, device=DEV)
    assert p.sense(y, cg_iters=2)[1].status == 0
    smsm.lib().smsm_plan_raise_for_test(p._h, smsm.SMSM_ERR_TIMEOUT)
    assert p.sense(y, cg_iters=2)[1].status == smsm.SMSM_ERR_TIMEOUT
    assert p.reconstruct(y)[1].status == smsm.SMSM_ERR_TIMEOUT
    assert p.device_status() == smsm.SMSM_ERR_TIMEOUT

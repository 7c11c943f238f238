"""Reverse mode reports a device wait that gave up (wait limit 0, as in test_gpu_faults): the calls
that hand out fields, states or derivatives return LBM_ERR_TIMEOUT, a sweep that gave up leaves the
parameter sums as they were, and a rerun gives the first run's bits."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu
TIMEOUT = -5


@pytest.fixture(scope="module")
def L():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2505_10899_gb300 import build
    build.build()
    from paper_2505_10899_gb300 import adjoint, lbm
    return lbm, adjoint


def _inputs():
    case = W.base_case(128, 64, sigma=4e-3, tau_f_l=0.9, tau_f_g=0.9)
    return case, W.tanh_disc(128, 64, 64.3, 32.2, 16, 4.0, True)


def test_sweep_timeout_is_reported_and_leaves_the_parameter_sums(L):
    import torch
    lbm, A = L
    case, phi0 = _inputs()
    a = A.AdjointSim(case, phi0, None, "f32")
    rec = torch.empty((8, a.planes) + a.shape, dtype=a.dtype, device="cuda")
    stride = rec[0].numel() * 4
    lbm.lbm_record_steps(a.h, 8, rec.data_ptr(), stride)
    lam = torch.ones((20, 64, 128), device="cuda")
    spare = torch.empty_like(lam)

    def sweep(n):
        x = lam.clone()
        lbm.lbm_adjoint_sweep(a.h, rec.data_ptr(), stride, 0, n, x.data_ptr(), spare.data_ptr())
        return x

    def take():
        g = np.zeros(6)
        a.take_grads(g)
        return g

    sweep(3)
    g3 = take()
    x8 = sweep(8)
    g8 = take()
    assert np.abs(g8).max() > 0
    sweep(3)  # accumulated before the sweep that gives up
    lbm.lbm_set_wait_limit(a.h, 0)
    sweep(8)
    with pytest.raises(lbm.LbmError) as e:
        take()
    assert e.value.status == TIMEOUT
    assert a.sim.status() == TIMEOUT and a.sim.status() == lbm.LBM_OK
    lbm.lbm_set_wait_limit(a.h, -1)
    assert np.array_equal(take(), g3)
    assert torch.equal(sweep(8), x8) and np.array_equal(take(), g8)
    a.close()


@pytest.mark.parametrize("call", ["fields", "get_state", "save"])
def test_forward_timeout_is_reported_where_the_state_is_read(L, call):
    lbm, _ = L
    case, phi0 = _inputs()
    s = lbm.Sim(case, phi0, None, precision="f32")
    lbm.lbm_set_wait_limit(s.h, 0)
    s.step(8)
    lbm.lbm_set_wait_limit(s.h, -1)
    with pytest.raises(lbm.LbmError) as e:
        getattr(s, call)()
    assert e.value.status == TIMEOUT
    assert s.status() == TIMEOUT  # reported until it is cleared here
    getattr(s, call)()
    s.close()


@pytest.mark.parametrize("where", ["lbm_record_steps", "lbm_adjoint_sweep"])
def test_coupled_run_raises(L, monkeypatch, where):
    import torch
    lbm, A = L
    case, phi0 = _inputs()
    inner = getattr(lbm, where)

    def limited(h, *args):
        lbm.lbm_set_wait_limit(h, 0)
        inner(h, *args)
        lbm.lbm_set_wait_limit(h, -1)

    monkeypatch.setattr(A.lbm, where, limited)
    p = torch.tensor(phi0, dtype=torch.float32, requires_grad=True)
    th = torch.tensor([case["sigma"], case["tau_g"], case["lambda"], case["tau_f_l"]],
                      requires_grad=True)
    with pytest.raises(lbm.LbmError):
        A.coupled_run(p, th, case, 12, precision="f32").sum().backward()

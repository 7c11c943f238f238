"""The chip-resident multi-step kernel (csrc/lbm_resident.cuh) against the register kernel, which
runs the same per-node arithmetic from global memory, and against the FP64 oracle: smallest and
ragged tiles, walls, the vortex, uneven batches, odd and even step counts, several launches, and
recorded states.

Tolerances: FP64 as everywhere (1e-12 against the oracle); FP32 against the register kernel as
between any two kernel instantiations (2e-6: they may contract multiply-adds differently)."""
import numpy as np
import pytest

import oracle
import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def L():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2505_10899_gb300 import build
    build.build()
    from paper_2505_10899_gb300 import lbm
    return lbm


def md(a, b):
    return 0.0 if a is None else float(np.abs(np.asarray(a) - np.asarray(b)).max())


def setup(nx, ny, kind, seed=3):
    if kind == "vortex":
        case = W.base_case(nx, ny, flow="vortex", W=3.0, sigma=0.01, vortex_U=0.02, vortex_T=90.0)
    else:
        kw = dict(walls=1, u_top=0.02, u_bot=-0.01) if kind == "walls" else {}
        case = W.base_case(nx, ny, sigma=5e-3, rho_l=3.0, tau_f_l=0.7, tau_f_g=1.1, **kw)
    return case, W.random_state(nx, ny, seed, coupled=kind != "vortex", phi_lo=0.05, phi_hi=0.95)


@pytest.mark.parametrize("kind", ["periodic", "walls", "vortex"])
@pytest.mark.parametrize("nx,ny", [(3, 3), (20, 3), (4, 9), (67, 5), (128, 64), (201, 101), (380, 190)])
@pytest.mark.parametrize("prec", ["f32", "f64"])
def test_matches_register_kernel_and_oracle(L, prec, nx, ny, kind):
    case, (f, g, j) = setup(nx, ny, kind)
    a = L.Sim(case, np.zeros((ny, nx)), None, precision=prec)
    b = L.Sim(case, np.zeros((ny, nx)), None, precision=prec)
    b.set_kernel(1)
    for s in (a, b):
        s.set_state(0, f, g, j, 4)
        for n in (5, 8, 4):  # odd and even counts, from either buffer
            s.step(n)
        assert s.t == 21 and s.status() == L.LBM_OK
    x, y = a.get_state(0), b.get_state(0)
    tol = 2e-6 if prec == "f32" else 1e-12
    for p, q in zip(x[:3], y[:3]):
        assert md(p, q) <= tol
    if prec == "f64" and nx * ny < 30000:
        o = oracle.Oracle(case, state=(f, g, j, 4)).step(17)
        assert md(x[0], o.f) <= 1e-12 if kind != "vortex" else True
        assert md(x[1], o.g) <= 1e-12 and md(x[2], o.j) <= 1e-12
    a.close(), b.close()


def test_more_steps_than_one_launch(L):
    # 2500 steps: three launches of up to 1024; the step clock (the vortex reads it) goes on
    case, phi0, _ = W.single_vortex(n=64, W=3.0, U=0.02, T=5000)
    out = []
    for k in (0, 1):
        s = L.Sim(case, phi0, None, precision="f32")
        s.set_kernel(k)
        s.step(2500)
        s.step(1)   # a direct step reads the device clock
        out.append(s.get_state(0))
        assert s.t == 2501 and s.status() == L.LBM_OK
        s.close()
    assert md(out[0][1], out[1][1]) <= 1e-5  # 2500 steps of FP32 rounding


def test_uneven_batch(L):
    specs = [(64, 64, 1.0), (192, 40, 4.0), (37, 52, 10.0), (4, 9, 2.0)]
    cases, phis = [], []
    for nx, ny, r in specs:
        cases.append(W.base_case(nx, ny, rho_l=r, walls=int(nx == 37)))
        phis.append(W.tanh_disc(nx, ny, nx / 2 + 0.3, ny / 2 + 0.2, min(nx, ny) / 4, 4.0, True))
    s = L.Sim(cases, phis, None, precision="f64")
    s.step(25)
    assert s.status() == L.LBM_OK
    for k, (c, p) in enumerate(zip(cases, phis)):
        o = oracle.Oracle(c, p).step(25)
        f, g, j, _ = s.get_state(k)
        assert md(f, o.f) <= 1e-12 and md(g, o.g) <= 1e-12 and md(j, o.j) <= 1e-12


@pytest.mark.parametrize("kind", ["walls", "vortex"])
@pytest.mark.parametrize("prec", ["f32", "f64"])
def test_recorded_states_are_the_snapshots(L, prec, kind):
    # lbm_record_steps in one launch: slot k holds lbm_snapshot of the state entering step k
    import torch
    nx, ny, n = 61, 40, 9
    case, (f, g, j) = setup(nx, ny, kind)
    dtype = torch.float32 if prec == "f32" else torch.float64
    planes = 21 if prec == "f32" else 20
    a = L.Sim(case, np.zeros((ny, nx)), None, precision=prec)
    a.set_state(0, f, g, j, 0)
    first = torch.empty((planes, ny, nx), dtype=dtype, device="cuda")
    L.lbm_snapshot(a.h, 0, first.data_ptr())
    rec = torch.full((n, planes, ny, nx), float("nan"), dtype=dtype, device="cuda")
    L.lbm_record_steps(a.h, n, rec.data_ptr(), rec[0].numel() * rec.element_size())
    assert a.t == n
    b = L.Sim(case, np.zeros((ny, nx)), None, precision=prec)
    b.set_kernel(1)
    b.set_state(0, f, g, j, 0)
    want = torch.empty_like(first)
    assert torch.equal(rec[0], first)
    tol = 2e-6 if prec == "f32" else 1e-12
    for k in range(n):
        L.lbm_snapshot(b.h, 0, want.data_ptr())
        assert float((rec[k] - want).abs().max()) <= tol, k
        b.step(1)
    assert a.status() == L.LBM_OK


@pytest.mark.parametrize("walls", [True, False], ids=["walls", "periodic"])
@pytest.mark.parametrize("nx,ny", [(20, 3), (67, 5), (128, 64), (201, 101), (512, 256)])
@pytest.mark.parametrize("count", [2, 9])
def test_reverse_sweep_matches_single_steps(L, nx, ny, walls, count):
    # one launch over recorded states against lbm_adjoint_step_from step by step.  The arithmetic
    # is the same up to the contraction of multiply-adds, an ulp (2^-23) of each of the sums that a
    # step adds up, tens of them: 1e-5 over nine steps.  Parameter sums differ in order as well.
    import torch
    from paper_2505_10899_gb300 import adjoint
    kw = dict(walls=1, u_top=0.02, u_bot=-0.01) if walls else {}
    case = W.base_case(nx, ny, sigma=5e-3, rho_l=2.0, tau_f_l=0.8, tau_f_g=0.8, **kw)
    phi0 = 0.5 + 0.3 * np.sin(np.arange(nx) * 2 * np.pi / nx)[None, :] * np.ones((ny, 1))
    phi0 = phi0 + W.uniform(4, (ny, nx), -0.1, 0.1)
    a = adjoint.AdjointSim(case, phi0, W.uniform(5, (2, ny, nx), -0.01, 0.01), "f32")
    a.step(3)
    rec = torch.empty((count, a.planes) + a.shape, dtype=a.dtype, device="cuda")
    L.lbm_record_steps(a.h, count, rec.data_ptr(), rec[0].numel() * 4)
    gen = torch.Generator(device="cuda").manual_seed(7)
    lam = torch.randn((20, ny, nx), generator=gen, device="cuda")
    got, spare = lam.clone(), torch.empty_like(lam)
    L.lbm_adjoint_sweep(a.h, rec.data_ptr(), rec[0].numel() * 4, 3, count, got.data_ptr(),
                        spare.data_ptr())
    g1, g2 = np.zeros(6), np.zeros(6)
    a.take_grads(g1)
    want = lam
    for j in range(count - 1, -1, -1):
        want = a.vjp_step_from(rec[j], 3 + j, want)
    a.take_grads(g2)
    assert a.sim.status() == L.LBM_OK
    assert float((got - want).norm() / want.norm()) <= 1e-5
    assert float((got - want).abs().max() / want.abs().max()) <= 1e-5
    assert np.abs(g1 - g2).max() <= 1e-4 * np.abs(g2).max()


def test_reverse_sweep_wait_limit(L):
    # at 0 cycles a CTA whose neighbours' rims have not come at its first poll gives up; the status
    # is reported once and the sweep runs again from its inputs
    import torch
    from paper_2505_10899_gb300 import adjoint
    case = W.base_case(128, 64)
    a = adjoint.AdjointSim(case, W.tanh_disc(128, 64, 64.3, 32.2, 16, 4.0, True), None, "f32")
    rec = torch.empty((8, a.planes) + a.shape, dtype=a.dtype, device="cuda")
    L.lbm_record_steps(a.h, 8, rec.data_ptr(), rec[0].numel() * 4)
    lam = torch.ones((20, 64, 128), device="cuda")
    out = []
    for limit in (-1, 0, -1):
        L.lbm_set_wait_limit(a.h, limit)
        x, spare = lam.clone(), torch.empty_like(lam)
        L.lbm_adjoint_sweep(a.h, rec.data_ptr(), rec[0].numel() * 4, 0, 8, x.data_ptr(),
                            spare.data_ptr())
        assert a.sim.status() == (L.LBM_ERR_TIMEOUT if limit == 0 else L.LBM_OK)
        out.append(x)
    assert torch.equal(out[0], out[2])

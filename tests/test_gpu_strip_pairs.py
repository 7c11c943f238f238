"""The strip kernel's two nodes per thread and chunk copies against the oracle where the shapes and
parameters differ from the general parity test: uniform relaxation time (no density ratio),
relaxation times above 2 (the complement 1 - 1/tau is rounded), many strips, one plane, no
sharpening, and runs long enough for graph replay.  Bars: those of the precision's parity tests."""
import numpy as np
import pytest

import oracle
import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec,bar", [("f32", 1e-5), ("f16", 2e-3)])
@pytest.mark.parametrize("variant,shape,tiling,kw", [
    (5, (320, 6, 9), (64, 4, 9), dict()),
    (6, (128, 4, 64), (64, 4, 64), dict(tau_f_l=2.7, tau_f_g=2.3, rho_l=2.0)),
    (6, (128, 7, 1), (64, 2, 1), {"lambda": 0.0}),
    (5, (64, 8, 2), (32, 8, 2), dict(tau_f_l=3.1, tau_f_g=3.1)),
])
def test_strip_pairs_against_oracle(variant, shape, tiling, kw, prec, bar):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2505_10899_gb300 import build
    build.build()
    from paper_2505_10899_gb300 import lbm3
    nx, ny, nz = shape
    case = W.base_case3(nx, ny, nz, **kw)
    x = np.arange(nx)[None, None, :]
    phi0 = np.ascontiguousarray(np.broadcast_to(
        0.5 * (1.0 + np.tanh(2.0 * (0.2 * nx - np.abs(x - 0.5 * nx + 0.3)) / 4.0)), (nz, ny, nx)))
    u0 = np.zeros((3, nz, ny, nx))
    u0[0], u0[1], u0[2] = 0.01, -0.005, 0.004
    s = lbm3.Sim3(case, phi0, u0, precision=prec)
    s.set_tiling(*tiling)
    s.set_kernel(variant)
    assert s.kernel() == variant and s.tiling()[:3] == tiling
    s.step(70)  # one replayed graph and single launches
    o = oracle.Oracle3(case, phi0, u0).step(70)
    assert s.status() == 0
    phi, u, _ = s.fields()
    ophi, ou, _ = o.fields()
    assert np.abs(phi - ophi).max() <= bar
    if prec == "f32":
        assert np.abs(u - ou).max() <= 1e-6
    assert abs(s.volume()[0] / phi0.sum() - 1) <= 1e-6
    s.close()

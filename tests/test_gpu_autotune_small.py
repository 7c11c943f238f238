"""Autotuning a batch that fits the chip: the chip-resident kernel is kept for the runs that it can
serve, and the tuned kernel and tile of single steps for the others (shorter runs, tracked volumes)."""
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


@pytest.mark.parametrize("nx,staged", [(128, True), (129, False)])
def test_small_batch_keeps_its_tuned_kernel(L, nx, staged):
    import torch
    case = W.base_case(nx, 64, rho_l=2.0)
    phi0 = W.tanh_disc(nx, 64, 64.3, 32.2, 16, 4.0, True)
    s = L.Sim(case, phi0, None, precision="f64")
    best = s.autotune(1)
    assert best["kernel"] in ((1, 2) if staged else (1,))
    assert s.kernel() == best["kernel"] and s.tiling()[:2] == (best["bx"], best["rows"])
    assert 1 <= s.resident() <= 4  # three times as fast and more at this size
    s.step(1)
    s.step(8)
    hist = s.track_volume_history(6, host=False)
    assert not s.resident()
    assert s.kernel() == best["kernel"] and s.tiling()[:2] == (best["bx"], best["rows"])
    s.step(6)  # slot t % 6 holds the volume at t = 9 .. 14
    torch.cuda.synchronize()
    o = oracle.Oracle(case, phi0).step(9)
    for t in range(9, 15):
        v = float(o.volume()[0])
        assert abs(float(hist[t % 6, 0]) - v) <= 1e-12 * v
        o.step(1)
    # tuned while tracking: nothing is tried that could not run
    assert s.autotune(1)["kernel"] in (1, 2) and not s.resident()
    s.track_volume(False)
    assert s.resident()
    f, g, j, t = s.get_state(0)
    assert t == 15
    assert max(np.abs(f - o.f).max(), np.abs(g - o.g).max(), np.abs(j - o.j).max()) <= 1e-12
    s.set_kernel(s.kernel())  # asked for: then it runs
    assert not s.resident()
    s.set_kernel(0)
    assert s.resident() == 4
    s.close()

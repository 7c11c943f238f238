"""lbm_autotune leaves a handle's state and its error flags alone: a state that is finite, but would
diverge a few steps later, tunes without an error and reads out as it was."""
import numpy as np
import pytest

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


@pytest.mark.parametrize("prec", ["f32", "f64"])
def test_autotune_before_a_divergence(L, prec):
    # a surface tension far beyond what is stable: phi overflows within ten steps
    case = W.base_case(128, 64, sigma=2.0)
    phi0 = W.tanh_disc(128, 64, 64.3, 32.2, 16, 4.0, True)
    s = L.Sim(case, phi0, None, precision=prec)
    before = s.get_state(0)
    s.autotune(1)
    v = s.volume()
    assert np.all(np.isfinite(v)) and s.status() == L.LBM_OK
    for a, b in zip(before[:3], s.get_state(0)[:3]):
        assert np.array_equal(a, b)
    s.step(64)  # it does diverge
    assert s.status() == L.LBM_ERR_NONFINITE
    s.close()

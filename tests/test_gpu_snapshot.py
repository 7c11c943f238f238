"""Device snapshots: the 16-byte and the one-value form write the same bits, and a snapshot
restored gives the state back.  Node counts that are and are not whole 16-byte groups, a target
that is and is not 16-byte aligned, both flows and precisions, two snapshots back to back."""
import numpy as np
import pytest
import torch

import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["f32", "f64"])
@pytest.mark.parametrize("flow", ["coupled", "vortex"])
@pytest.mark.parametrize("shape", [(128, 64), (201, 101), (66, 5), (4, 3)])
def test_snapshot_forms_agree(shape, flow, precision):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2505_10899_gb300 import build
    build.build()
    from paper_2505_10899_gb300 import lbm
    nx, ny = shape
    case = W.base_case(nx, ny, flow=flow)
    phi0 = W.tanh_disc(nx, ny, nx / 2 + 0.2, ny / 2 + 0.1, 0.25 * min(nx, ny), 4.0, periodic=True)
    s = lbm.Sim(case, phi0, None, precision=precision)
    s.step(3)
    dtype = torch.float32 if precision == "f32" else torch.float64
    n = lbm.lbm_snapshot_bytes(s.h, 0) // dtype.itemsize
    buf = torch.full((2 * n + 1,), 7.0, dtype=dtype, device="cuda")
    a, b = buf[:n], buf[n + 1:]  # one of the two starts off a 16-byte boundary
    lbm.lbm_snapshot(s.h, 0, a.data_ptr())
    lbm.lbm_snapshot(s.h, 0, b.data_ptr())
    assert torch.equal(a, b) and float(buf[n]) == 7.0
    before = s.get_state(0)
    s.step(5)
    lbm.lbm_restore(s.h, 0, b.data_ptr())
    for x, y in zip(before[:3], s.get_state(0)[:3]):
        assert x is None or np.array_equal(x, y)
    s.close()

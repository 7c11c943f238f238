"""Phase volumes in one launch (few work items) and in two, against FP64 host sums of the state:
both sides of the limit of items, one and many regions, nodes without a region, repeated calls
(the ticket word is reset), and the error flag that travels with the volumes."""
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
@pytest.mark.parametrize("nx,ny,tiling", [(5, 3, None), (128, 64, None), (256, 256, (32, 2)),
                                          (256, 258, (32, 2)), (700, 300, None)],
                         ids=["5x3", "128x64", "1024-items", "1032-items", "700x300"])
@pytest.mark.parametrize("nreg", [1, 3, 8])
def test_volumes_match_host_sums(L, prec, nx, ny, tiling, nreg):
    s = L.Sim(W.base_case(nx, ny), W.uniform(7, (ny, nx), 0.0, 1.0), None, precision=prec)
    if tiling:
        s.set_tiling(*tiling)
    s.step(1)
    lab = None
    if nreg > 1:
        lab = (W.splitmix64(5, nx * ny) % np.uint64(nreg + 1)).astype(np.int8).reshape(ny, nx) - np.int8(1)
        s.set_regions(0, lab, nreg)
    phi = s.get_state(0)[1].sum(0)
    want = np.array([phi.sum()] if lab is None else [phi[lab == r].sum() for r in range(nreg)])
    for _ in range(3):
        assert np.all(np.abs(s.volume() - want) <= 1e-13 * np.abs(phi).sum())
    s.close()


def test_volume_reports_nonfinite_state(L):
    phi0 = np.full((8, 8), 0.5)
    phi0[3, 3] = np.nan
    s = L.Sim(W.base_case(8, 8), phi0, None, precision="f32")
    s.step(1)
    with pytest.raises(L.LbmError) as e:
        s.volume()
    assert e.value.status == L.LBM_ERR_NONFINITE
    assert s.status() == L.LBM_ERR_NONFINITE

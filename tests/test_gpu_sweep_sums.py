"""Parameter sums of the chip-resident reverse sweep: at most 32 nodes' terms meet in FP32, as in
the single adjoint steps; above that they are FP64.  A thread of a full tile holds two nodes, 512
apart in the tile.  Adjoints are put on two small patches that far apart, the second 1e-4 of the
first: its terms share the first one's warps but no FP32 sum with it, so the derivatives of both
together are the sum of the derivatives of either (the sweep is linear, every other term an exact
zero) up to the FP64 rounding of a few hundred partial sums (1e-16 each, bar 1e-12).  In one FP32
sum the second would be rounded at 6e-8 of the first."""
import numpy as np
import pytest

import workloads as W
from test_resident_plan import plan  # noqa: F401  (the library's tiling, compiled for the host)

pytestmark = pytest.mark.gpu


def test_two_nodes_of_a_thread_do_not_share_an_fp32_sum(plan):  # noqa: F811
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2505_10899_gb300 import build
    build.build()
    from paper_2505_10899_gb300 import adjoint, lbm
    nx, ny = 512, 256
    tiles, _, (nt, r, *_) = plan([(nx, ny)], "f32", adjoint=1)
    assert (nt, r) == (512, 2)
    # a tile with room for patches of radius 4 in both halves (two adjoint steps reach 4 nodes)
    for _, x0, y0, w, h, *_ in tiles:
        spots = [(k % w, k // w) for k in range(nt)]
        good = [(x, y) for x, y in spots
                if 4 <= x < w - 4 and 4 <= y and (y + 4) * w + x + 4 < nt
                and 4 <= (y * w + x + nt) % w < w - 4
                and (y * w + x + nt) // w - 4 >= y + 5 and (y * w + x + nt) // w + 4 < h]
        if good:
            break
    ax, ay = good[len(good) // 2]
    bx, by = (ay * w + ax + nt) % w, (ay * w + ax + nt) // w
    case = W.base_case(nx, ny, sigma=5e-3, rho_l=2.0, tau_f_l=0.8, tau_f_g=0.8)
    phi0 = 0.5 + W.uniform(4, (ny, nx), -0.2, 0.2)
    a = adjoint.AdjointSim(case, phi0, W.uniform(5, (2, ny, nx), -0.01, 0.01), "f32")
    a.step(2)
    rec = torch.empty((2, a.planes) + a.shape, device="cuda")
    a.record(rec)
    lam = W.uniform(9, (2, 20), 0.5, 1.0)

    def grads(sa, sb):
        adj = a.new_state()
        adj[:, y0 + ay, x0 + ax] = torch.as_tensor(sa * lam[0], dtype=torch.float32)
        adj[:, y0 + by, x0 + bx] = torch.as_tensor(sb * lam[1], dtype=torch.float32)
        a.sweep(rec, 0, adj, torch.empty_like(adj))
        g = np.zeros(6)
        a.take_grads(g)
        return g[:4]

    ga, gb, gab = grads(1.0, 0.0), grads(0.0, 1e-4), grads(1.0, 1e-4)
    assert a.sim.status() == lbm.LBM_OK
    assert np.abs(gb).min() > 0
    assert np.all(np.abs(gab - ga - gb) <= 1e-12 * np.abs(ga).max()), (ga, gb, gab - ga - gb)
    a.close()

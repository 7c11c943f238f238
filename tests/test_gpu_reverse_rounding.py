"""FP64 reverse mode keeps one rounding of the forward step.

d psi / d phi is up to 1/xi = 1e10 in the bulk, so the derivatives of a run move by up to 1e-8 when
the last bits of its states do.  A handle with reverse mode attached therefore steps by division,
root and logarithm and the general collision (lbm_handle::plain), and every route to a state gives
the bits of the single-step kernel.

The recorded values are those of the library before its FP64 step had shorter forms (reciprocal and
logarithm of lbm_math.cuh, collision at unit rates).  The runs below are among those that show a
rounding most: with the shorter forms they come out 2.5e-8, 4.5e-9 and 8.6e-9 away.  Bar 1e-12.  The initial fields
are made of additions, products, quotients and square roots only, which every machine rounds alike."""
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
    from paper_2505_10899_gb300 import adjoint, lbm
    return lbm, adjoint


def disc(nx, ny, cx, cy, R, width):
    x = np.arange(nx, dtype=np.float64)[None, :] - cx
    y = np.arange(ny, dtype=np.float64)[:, None] - cy
    s = np.clip((R - np.sqrt(x * x + y * y)) / width, -1.0, 1.0)
    return 0.5 + s * (15.0 - s * s * (10.0 - 3.0 * s * s)) * 0.0625


# nx, ny, profile width, seed, steps: d/d(sigma, tau_g, lambda, tau_f), and d/dphi0 at one node
GOLDEN = [
    (96, 80, 4.0, 29, 24, [9.101981667642288, -0.36739648707020645, -0.28119286274604605,
                           0.0003380458243715161], (3519, -34966.030127691745)),
    (128, 64, 3.0, 10, 32, [-12.673939332986441, 0.3892948491885409, 0.22085244469434429,
                            -0.0001425423647714555], (3394, 147.87567346043977)),
    (64, 48, 4.0, 9, 24, [-7.539114232890193, 0.3597302999333686, 0.29115362652280474,
                          -0.0006693362909087246], (1889, 12533.139903564137)),
]


@pytest.mark.parametrize("nx,ny,width,seed,steps,dtheta,dphi", GOLDEN)
def test_fp64_gradient_keeps_its_values(L, nx, ny, width, seed, steps, dtheta, dphi):
    import torch
    _, A = L
    r = W.uniform(seed, (6,), 0.0, 1.0)
    case = W.base_case(nx, ny, sigma=5e-3, tau_f_l=0.9, tau_f_g=0.9)
    phi0 = disc(nx, ny, nx / 2 + r[0], ny / 2 + r[1], (0.15 + 0.1 * r[2]) * min(nx, ny), width)
    u0 = np.zeros((2, ny, nx))
    u0[0], u0[1] = 0.005 + 0.005 * r[3], 0.01 * r[4] - 0.005
    w = torch.as_tensor(W.uniform(seed + 100, (ny, nx), 0.0, 1.0), device="cuda")
    p = torch.tensor(phi0, requires_grad=True)
    th = torch.tensor([case["sigma"], case["tau_g"], case["lambda"], case["tau_f_l"]],
                      dtype=torch.float64, requires_grad=True)
    phi = A.coupled_run(p, th, case, steps, u0=u0)
    gp, gt = torch.autograd.grad((phi * w).sum(), (p, th))
    want = np.array(dtheta)
    assert np.all(np.abs(gt.numpy() - want) <= 1e-12 * np.abs(want)), (gt.tolist(), dtheta)
    got = gp.flatten()[dphi[0]].item()
    assert abs(got - dphi[1]) <= 1e-12 * abs(dphi[1]), (got, dphi[1])


@pytest.mark.parametrize("kind", ["periodic", "walls", "vortex"])
@pytest.mark.parametrize("nx,ny", [(4, 3), (66, 40), (128, 64), (97, 65), (256, 160), (401, 251)])
def test_recorded_states_have_the_bits_of_single_steps(L, nx, ny, kind):
    # staged and register kernels, both sizes of the chip-resident kernel and grids beyond it
    import torch
    lbm, A = L
    if kind == "vortex":
        case = W.base_case(nx, ny, flow="vortex", W=3.0, sigma=0.01, vortex_U=0.02, vortex_T=90.0)
    else:
        kw = dict(walls=1, u_top=0.02, u_bot=-0.01) if kind == "walls" else {}
        case = W.base_case(nx, ny, sigma=5e-3, rho_l=3.0, tau_f_l=0.7, tau_f_g=1.1, **kw)
    phi0 = disc(nx, ny, 0.5 * nx + 0.3, 0.5 * ny + 0.2, 0.3 * min(nx, ny), 4.0)
    n = 6
    a, b = (A.AdjointSim(case, phi0) for _ in range(2))
    rec = torch.empty((n, a.planes, ny, nx), dtype=torch.float64, device="cuda")
    lbm.lbm_record_steps(a.h, n, rec.data_ptr(), rec[0].numel() * 8)
    for k in range(n):
        assert torch.equal(rec[k], b.snapshot()), k
        b.step(1)
    assert torch.equal(a.snapshot(), b.snapshot())
    a.close(), b.close()

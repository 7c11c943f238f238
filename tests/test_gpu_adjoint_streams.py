"""Reverse mode called from another stream than the handle's, with either stream busy: the results
are those of one stream, bit for bit."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["f32", "f64"])
@pytest.mark.parametrize("busy", ["caller", "handle"])
def test_side_stream_gives_the_same_bits(prec, busy):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2505_10899_gb300 import build
    build.build()
    from paper_2505_10899_gb300 import adjoint
    case = W.base_case(64, 48, rho_l=2.0, tau_f_l=0.9, tau_f_g=0.9)
    phi0 = W.tanh_disc(64, 48, 31.3, 24.2, 12, 4.0, True)

    def run(side):
        cur = torch.cuda.current_stream()
        with torch.cuda.stream(side):
            a = adjoint.AdjointSim(case, phi0, None, prec)
        cur.wait_stream(side)
        slow = cur if (busy == "caller" or side == cur) else side

        def delay():  # about 10 ms of work that the other stream does not wait for by itself
            with torch.cuda.stream(slow):
                torch.cuda._sleep(20_000_000)

        out = []
        for call in (lambda: a.phi(), lambda: a.snapshot(),
                     lambda: a.seed_phi(torch.full((48, 64), 0.5, device="cuda")),
                     lambda: a.vjp_step(torch.ones_like(a.new_state())),
                     lambda: a.vjp_init(torch.ones_like(a.new_state()), None)):
            delay()
            out.append(call().clone())
        rec = torch.zeros((4, a.planes) + a.shape, dtype=a.dtype, device="cuda")
        delay()
        a.record(rec)
        adj = torch.ones_like(a.new_state())
        delay()
        a.sweep(rec, 0, adj, torch.empty_like(adj))
        out += [rec.clone(), adj.clone()]
        delay()
        a.restore(rec[1].clone(), 1)
        out.append(a.vjp_step_from(rec[2].clone(), 2, adj.clone()).clone())
        out.append(a.snapshot().clone())
        g = np.zeros(6)
        a.take_grads(g)
        out.append(torch.as_tensor(g))
        torch.cuda.synchronize()
        a.close()
        return out

    want = run(torch.cuda.current_stream())
    got = run(torch.cuda.Stream())
    for k, (x, y) in enumerate(zip(want, got)):
        assert torch.equal(x, y), k

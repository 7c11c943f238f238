"""Order between a reverse-mode handle's stream and its caller's, on the CPU: every method that
hands tensors to the library makes the handle's stream wait for the caller's before the call and
the caller's wait for the handle's after it, and creates or fills no tensor of the call between."""
import contextlib
import types

import pytest
import torch

from paper_2505_10899_gb300 import adjoint

LIBRARY = ("lbm_snapshot", "lbm_restore", "lbm_set_time", "lbm_field_phi", "lbm_adjoint_seed_phi",
           "lbm_adjoint_step", "lbm_adjoint_step_from", "lbm_adjoint_init", "lbm_record_steps",
           "lbm_adjoint_sweep")


class Stream:
    def __init__(self, name, log):
        self.name, self.log = name, log

    def wait_stream(self, other):
        self.log.append((self.name, "waits for", other.name))


@pytest.fixture
def asim(monkeypatch):
    log = []
    cur, own = Stream("caller", log), Stream("handle", log)
    monkeypatch.setattr(torch.cuda, "current_stream", lambda dev=None: cur)
    for name in LIBRARY:
        def call(*args, _n=name):
            if _n != "lbm_set_time":  # host state only
                log.append(("library", _n))
            return adjoint.lbm.LBM_OK
        monkeypatch.setattr(adjoint.lbm, name, call)
    a = object.__new__(adjoint.AdjointSim)
    a.sim = types.SimpleNamespace(stream=own)
    a.h, a.dev, a.dtype, a.shape, a.planes = 1, torch.device("cpu"), torch.float64, (4, 6), 20
    a.phi0, a.u0 = torch.zeros(a.shape, dtype=torch.float64), None
    for fill in ("empty", "zeros"):
        inner = getattr(torch, fill)

        def make(*args, _f=inner, **kw):
            log.append(("caller", "makes a tensor"))
            return _f(*args, **kw)
        monkeypatch.setattr(adjoint.torch, fill, make)
    return a, log, cur, own


STATE = torch.ones((3, 20, 4, 6), dtype=torch.float64)
CALLS = {
    "snapshot": lambda a: a.snapshot(),
    "restore": lambda a: a.restore(STATE[0], 3),
    "phi": lambda a: a.phi(),
    "seed_phi": lambda a: a.seed_phi(torch.ones(4, 6)),
    "vjp_step": lambda a: a.vjp_step(STATE[0]),
    "vjp_step_from": lambda a: a.vjp_step_from(STATE[0], 2, STATE[1]),
    "vjp_init": lambda a: a.vjp_init(STATE[0], None),
    "record": lambda a: a.record(STATE),
    "sweep": lambda a: a.sweep(STATE, 0, STATE[0], STATE[1]),
}


@pytest.mark.parametrize("name", sorted(CALLS))
def test_both_streams_wait(asim, name):
    a, log, _, _ = asim
    CALLS[name](a)
    at = [k for k, e in enumerate(log) if e[0] == "library"]
    assert len(at) == 1, log
    assert log[at[0] - 1] == ("handle", "waits for", "caller"), log
    assert log[at[0] + 1:] == [("caller", "waits for", "handle")], log


@pytest.mark.parametrize("name", sorted(CALLS))
def test_one_stream_needs_no_wait(asim, name, monkeypatch):
    a, log, cur, _ = asim
    a.sim.stream = cur
    CALLS[name](a)
    assert not [e for e in log if e[1] == "waits for"]


def test_the_caller_waits_after_an_error(asim, monkeypatch):
    a, log, _, _ = asim

    def fails(*args):
        log.append(("library", "fails"))
        raise adjoint.lbm.LbmError(-1, "x", "y")
    monkeypatch.setattr(adjoint.lbm, "lbm_snapshot", fails)
    with contextlib.suppress(adjoint.lbm.LbmError):
        a.snapshot()
    assert log[-1] == ("caller", "waits for", "handle")

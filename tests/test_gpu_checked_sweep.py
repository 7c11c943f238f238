"""The chip-resident reverse sweep and recording under the debug build with index checks: no index
flag on ragged tiles, walls and full tiles, and the derivatives of the single adjoint steps (the
bars of test_gpu_resident).  The checked library is loaded in a child process.  On the CPU: in that
build's source every global access of the sweep kernel is behind a check."""
import os
import re
import subprocess
import sys

import pytest

from conftest import ROOT

SCRIPT = r'''
import sys
import numpy as np, torch
sys.path.insert(0, ROOT)
import workloads as W
from paper_2505_10899_gb300 import adjoint, lbm
assert lbm.LIB_PATH.endswith("liblbm_gb300_checked.so")
for nx, ny, walls in ((20, 3, 0), (67, 5, 1), (201, 101, 1), (128, 64, 0), (512, 256, 1)):
    case = W.base_case(nx, ny, sigma=5e-3, rho_l=2.0, tau_f_l=0.8, tau_f_g=0.8, walls=walls)
    phi0 = 0.5 + W.uniform(4, (ny, nx), -0.2, 0.2)
    a = adjoint.AdjointSim(case, phi0, None, "f32")
    rec = torch.empty((5, a.planes) + a.shape, device="cuda")
    a.record(rec)
    lam = torch.randn((20, ny, nx), generator=torch.Generator(device="cuda").manual_seed(7),
                      device="cuda")
    got = lam.clone()
    a.sweep(rec, 0, got, torch.empty_like(lam))
    g1, g2 = np.zeros(6), np.zeros(6)
    a.take_grads(g1)
    want = lam
    for j in range(4, -1, -1):
        want = a.vjp_step_from(rec[j], j, want)
    a.take_grads(g2)
    assert a.sim.status() == lbm.LBM_OK, (nx, ny)
    assert float((got - want).norm() / want.norm()) <= 1e-5
    assert np.abs(g1 - g2).max() <= 1e-4 * np.abs(g2).max()
    a.close()
print("checked ok")
'''


@pytest.mark.gpu
def test_checked_sweep_raises_no_index_flag():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2505_10899_gb300 import build
    build.build(checked=True)
    env = dict(os.environ, LBM_GB300_CHECKED="1")
    r = subprocess.run([sys.executable, "-c", f"ROOT = {ROOT!r}\n" + SCRIPT], cwd=ROOT, env=env,
                       capture_output=True, text=True, timeout=900)
    assert r.returncode == 0 and "checked ok" in r.stdout, r.stdout[-2000:] + r.stderr[-3000:]


def test_every_global_access_of_the_sweep_is_checked():
    src = open(os.path.join(ROOT, "paper_2505_10899_gb300", "csrc",
                            "lbm_adjoint_resident.cuh")).read()
    body = re.sub(r"//[^\n]*", "", src[src.index("ad_resident("):])
    # the check that covers an access stands in the same loop body, before it or on its line
    lines = body.split("\n")
    access = {r"\b[fg]A \+ p \* n \+ pos": r"pos, n\)", r"\bJA \+": r"node, n\)",
              r"run\.adj\[": r"node, n\)", r"run\.slots \+": r"[de]\.x, run\.nslots\)",
              r"prefetch\.global": r"at, 20 \* "}
    seen = 0
    for k, line in enumerate(lines):
        for pat, check in access.items():
            if re.search(pat, line):
                seen += 1
                near = "\n".join(lines[max(0, k - 32):k + 1])
                assert re.search(r"LBM_BOUND\(run\.flags, " + check, near), (k, line)
    assert seen >= 12
    # a full rim table is flagged, and not read beyond its end
    assert body.count("else\n      atomicOr(run.flags, lbmk::kFlagBounds)") == 2
    assert "min(nrecv_s, kAdNX)" in body and "min(nsend_s, kAdNX)" in body

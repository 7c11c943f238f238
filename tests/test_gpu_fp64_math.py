"""FP64 reciprocal, reciprocal square root and log ratio of csrc/lbm_math.cuh on the GPU, against
extended-precision host values.  Bounds from their construction: one third-order step from 20
bits leaves 2^-58 before rounding (2 ulp in all); the logarithm's table entries, ln 2 and sums
round to half an ulp each (|error| <= 3e-16 + 2.5e-16 |ln(a/b)|).  Arguments with zero, subnormal,
infinite or NaN parts take CUDA's log."""
import ctypes
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

SRC = r'''
#include "lbm_math.cuh"
__global__ void k(const double* a, const double* b, double* o, int n) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  o[i] = lbmk::rcp64(a[i]);
  o[n + i] = lbmk::rsq64(a[i]);
  o[2 * n + i] = lbmk::lratio64(a[i], b[i]);
}
extern "C" int run(const double* a, const double* b, double* o, int n) {
  k<<<(n + 255) / 256, 256>>>(a, b, o, n);
  return (int)cudaDeviceSynchronize();
}
'''


@pytest.fixture(scope="module")
def gpu_math(tmp_path_factory):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2505_10899_gb300 import build
    d = tmp_path_factory.mktemp("math")
    (d / "m.cu").write_text(SRC)
    subprocess.run([build.nvcc(), *build._flags(), "-shared", str(d / "m.cu"), "-o", str(d / "m.so")],
                   check=True)
    lib = ctypes.CDLL(str(d / "m.so"))

    def call(a, b):
        ta, tb = (torch.from_numpy(np.ascontiguousarray(v)).cuda() for v in (a, b))
        out = torch.empty((3, len(a)), dtype=torch.float64, device="cuda")
        torch.cuda.synchronize()
        rc = lib.run(*(ctypes.c_void_p(t.data_ptr()) for t in (ta, tb, out)), len(a))
        assert rc == 0
        return out.cpu().numpy()
    return call


def test_rcp_rsq_within_two_ulp(gpu_math):
    rng = np.random.default_rng(1)
    x = np.concatenate([np.exp(rng.uniform(-40, 40, 200000)), 1.0 + rng.uniform(-1e-12, 1e-12, 1000),
                        2.0 ** np.arange(-60, 60), np.nextafter(2.0 ** np.arange(-60, 60), 0)])
    r, s, _ = gpu_math(x, np.ones_like(x))
    xl = x.astype(np.longdouble)
    for got, want in ((r, 1 / xl), (s, 1 / np.sqrt(xl))):
        assert float(np.max(np.abs(got - want) / np.spacing(want.astype(np.float64)))) <= 2.0


def test_log_ratio(gpu_math):
    rng = np.random.default_rng(2)
    xi = 1e-10
    phi = np.concatenate([rng.uniform(0, 1, 200000), 1e-10 * rng.uniform(0, 10, 1000),
                          1 - 1e-10 * rng.uniform(0, 10, 1000), [0.0, 1.0, 0.5],
                          (np.arange(1, 512) / 512.0)])
    a, b = phi + xi, (1.0 - phi) + xi
    got = gpu_math(a, b)[2]
    want = np.log(a.astype(np.longdouble)) - np.log(b.astype(np.longdouble))
    bound = 3e-16 + 2.5e-16 * np.abs(want).astype(np.float64)
    assert np.all(np.abs(got - want).astype(np.float64) <= bound)
    # special arguments: as log(a / b)
    a = np.array([0.0, 1.0, np.inf, np.nan, 1.0, 5e-310, -1.0])
    b = np.array([1.0, 0.0, 1.0, 1.0, np.nan, 1.0, 1.0])
    with np.errstate(all="ignore"):
        want = np.log(a / b)
    assert np.allclose(gpu_math(a, b)[2], want, rtol=1e-15, equal_nan=True)

"""The FP64 form's exp, log and quotient against 64-bit numpy, at the edges of their ranges."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2010_14823_gb300 import build  # noqa: E402

pytestmark = pytest.mark.gpu

_SRC = r"""
#include "casim_math64.cuh"
__global__ void k(const double *a, const double *b, double *o, int n) {
  const int i = blockIdx.x * 256 + threadIdx.x;
  if (i >= n) return;
  o[i] = casim_dev::exp64(a[i]);
  o[n + i] = casim_dev::log64(b[i]);
  o[2 * n + i] = casim_dev::div64(a[i], b[i]);
}
extern "C" int run(const double *a, const double *b, double *o, int n) {
  k<<<(n + 255) / 256, 256>>>(a, b, o, n);
  return (int)cudaDeviceSynchronize();
}
"""


@pytest.fixture(scope="module")
def run(tmp_path_factory):
    d = tmp_path_factory.mktemp("math64")
    (d / "m.cu").write_text(_SRC)
    so = os.path.join(d, "m.so")
    subprocess.run([build.nvcc()] + build.NVCC_FLAGS + ["-I" + build.CSRC, "-shared", "-o", so, str(d / "m.cu")], check=True)
    lib = ctypes.CDLL(so)

    def f(a, b):
        ta, tb = torch.from_numpy(a).cuda(), torch.from_numpy(b).cuda()
        o = torch.empty((3, len(a)), dtype=torch.float64, device="cuda")
        ptr = lambda t: ctypes.c_void_p(t.data_ptr())  # noqa: E731
        assert lib.run(ptr(ta), ptr(tb), ptr(o), len(a)) == 0
        return o.cpu().numpy()
    return f


def test_accuracy_and_special_values(run):
    """Each within 1.5 ulp of numpy's (which is itself within 1 ulp: 2.5 ulp); special values equal."""
    rng = np.random.default_rng(2)
    a = np.concatenate([rng.uniform(-700.5, 700.5, 20000), rng.uniform(-1e-3, 1e-3, 5000), [0.0, -0.0, 699.99, 700.0, -745.0]])
    b = np.concatenate([np.exp(rng.uniform(-700, 700, 20000)), 1 + rng.uniform(-0.02, 0.02, 5000),
                        [1.0, 2.0, 0.5, 2.2250738585072014e-308, 5e-324]])
    got = run(a, b)
    with np.errstate(over="ignore", under="ignore"):
        want = np.exp(a), np.log(b), a / b
    for g, w in zip(got, want):
        ok = np.isfinite(w) & (np.abs(w) > 1e-300)
        assert (np.abs(g[ok] - w[ok]) <= 2.5 * np.spacing(np.abs(w[ok]))).all()
        assert np.array_equal(np.isinf(g), np.isinf(w))
    special = np.array([0.0, -0.0, np.inf, -np.inf, np.nan, 800.0, -800.0, -1.0])
    x, y = (v.ravel().copy() for v in np.meshgrid(special, special))
    got = run(x, y)
    with np.errstate(all="ignore"):
        for g, w in zip(got, (np.exp(x), np.log(y), x / y)):
            ok = np.isfinite(w) & (w != 0)
            assert np.array_equal(g[~ok], w[~ok], equal_nan=True)
            assert np.allclose(g[ok], w[ok], rtol=1e-15, atol=0)

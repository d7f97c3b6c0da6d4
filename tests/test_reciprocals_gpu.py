"""The reciprocal and the short reciprocal square root that the solvers' chains are made of,
compiled from the library's own header: over the exponent range and where they change branch."""
import ctypes
import pathlib
import shutil
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

CSRC = pathlib.Path(__file__).resolve().parent.parent / "paper_2601_19650_gb300" / "csrc"
SOURCE = """
#include "common.cuh"
__global__ void k(const double* x, double* r, double* s, int n) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) {
    r[i] = cbc::rcp64(x[i]);
    s[i] = x[i] > 0.0 ? cbc::rsqrt64_short(x[i]) : 0.0;
  }
}
extern "C" void run(const double* x, double* r, double* s, int n) {
  k<<<(n + 255) / 256, 256>>>(x, r, s, n);
}
"""


def _near(a, b, ulps):
    """|a - b| in units of the last place of b, subnormal results to their absolute spacing"""
    return np.all(np.abs(a - b) <= ulps * np.spacing(np.abs(b)))


def test_over_the_exponent_range(tmp_path):
    import torch
    (tmp_path / "k.cu").write_text(SOURCE)
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    subprocess.run([nvcc, "-gencode", "arch=compute_103a,code=sm_103a", "-O3", "-std=c++17",
                    "-shared", "-Xcompiler", "-fPIC", f"-I{CSRC}", "-o", str(tmp_path / "k.so"),
                    str(tmp_path / "k.cu")], check=True)
    run = ctypes.CDLL(str(tmp_path / "k.so")).run
    rng = np.random.default_rng(1)
    # every exponent, and mantissas at and next to its ends
    e = np.arange(-1022, 1024)
    m = np.concatenate([rng.uniform(1, 2, 20), [1.0, np.nextafter(1, 2), np.nextafter(2, 1), 1.5]])
    x = np.concatenate([np.ldexp(m[None, :], e[:, None]).ravel(),
                        np.ldexp(rng.integers(1, 2 ** 52, 200).astype(float), -1074),
                        [5e-324, 2.0 ** -1022, np.nextafter(2.0 ** -1022, 0)]])
    x = np.concatenate([x, -x])
    d = torch.from_numpy(x).cuda()
    r, s = torch.zeros_like(d), torch.zeros_like(d)
    torch.cuda.synchronize()
    run(*(ctypes.c_void_p(t.data_ptr()) for t in (d, r, s)), len(x))
    torch.cuda.synchronize()
    r, s = r.cpu().numpy(), s.cpu().numpy()
    with np.errstate(over="ignore"):
        want = (1 / x.astype(np.longdouble)).astype(float)
    fin = np.isfinite(want)
    assert np.array_equal(np.isinf(r), ~fin)
    # a 20-bit start and one cubic step: the rounding of the step's own two operations
    assert _near(r[fin], want[fin], 1)
    pos = x > 0
    assert _near(s[pos], (1 / np.sqrt(x[pos].astype(np.longdouble))).astype(float), 2)

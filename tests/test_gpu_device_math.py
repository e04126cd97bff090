"""The kernels' own arithmetic (k_m2l.cuh), value by value against numpy over the ranges that the kernels use, through
a small library compiled around the header.  Tolerances: the roundings of each function counted at its test."""
import ctypes
import subprocess

import numpy as np
import pytest

from paper_2306_11324_gb300 import build

pytestmark = pytest.mark.gpu

SOURCE = r"""
#include "k_m2l.cuh"

using namespace igabem;

__global__ void k_eval(int what, long n, const double *a, const double *b, const double *c, double *out) {
  const long i = blockIdx.x * (long)blockDim.x + threadIdx.x;
  if (i >= n) return;
  if (what == 0) out[i] = phase32((float)a[i], (float)b[i], (float)c[i]);
}

// device arrays of n values
extern "C" int eval(int what, long n, const double *a, const double *b, const double *c, double *out) {
  k_eval<<<(unsigned)((n + 255) / 256), 256>>>(what, n, a, b, c, out);
  const cudaError_t e = cudaDeviceSynchronize();
  return (int)e;
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("math")
    (d / "eval.cu").write_text(SOURCE)
    so = d / "libeval.so"
    subprocess.run([build._nvcc(), "-shared", str(d / "eval.cu"), "-o", str(so)] + build.ARCH + build.FLAGS, check=True)
    L = ctypes.CDLL(str(so))
    L.eval.argtypes = [ctypes.c_int, ctypes.c_long] + [ctypes.c_void_p] * 4
    return L


def evaluate(lib, what, outputs, *args):
    import torch
    n = len(args[0])
    t = [torch.from_numpy(np.ascontiguousarray(x, dtype=np.float64)).cuda() for x in args]
    t += [torch.zeros(1, dtype=torch.float64, device="cuda")] * (3 - len(t))
    out = torch.empty((outputs, n), dtype=torch.float64, device="cuda")
    torch.cuda.synchronize()
    assert lib.eval(what, n, *[x.data_ptr() for x in t], out.data_ptr()) == 0
    return out.cpu().numpy()


@pytest.mark.parametrize("kappa", [0.0, 0.3, 5.0, 11.0, 27.0, 250.0])
def test_phase32(lib, kappa):
    """kappa d + phi0 modulo 2 pi: the sum rounds to half a unit in its last place (2^-24 of it), the two steps of the
    reduction to half a unit of pi each (2^-23)."""
    rng = np.random.default_rng(int(kappa))
    kappa = float(np.float32(kappa))
    d = np.float32(rng.uniform(-0.5, 0.5, 100_000)).astype(float)
    phi0 = np.float32(rng.uniform(-np.pi, np.pi, d.size)).astype(float)
    got = evaluate(lib, 0, 1, np.full(d.size, kappa), d, phi0)[0]
    exact = kappa * d + phi0
    error = np.mod(got - exact + np.pi, 2 * np.pi) - np.pi
    assert np.abs(got).max() < 3.2
    assert (np.abs(error) <= 2.0 ** -24 * np.abs(exact) + 2 * 2.0 ** -23 + 1e-12).all()

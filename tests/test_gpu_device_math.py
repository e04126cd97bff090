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
  if (what == 1) out[i] = rsqrt64(a[i]);
  if (what == 2) out[i] = rcp64(a[i]);
  if (what == 3) {  // exp(i kappa r), the table in c
    double c0, c1;
    phase64_scale(a[i], c0, c1);
    const Phase64 p = phase64(reinterpret_cast<const double2 *>(c), b[i], c0, c1);
    const C2<double> v = phase_mul(p.E.x, p.E.y, p);
    out[i] = v.x;
    out[n + i] = v.y;
  }
  if (what == 4) {
    float s, cm;
    sin_cosm1((float)a[i], s, cm);
    out[i] = s;
    out[n + i] = cm;
  }
  if (what == 5) {
    float s = (float)a[i], l = 0.f;
    two_sum(s, l, (float)b[i]);
    two_sum(s, l, (float)c[i]);
    out[i] = (double)s + (double)l;
  }
}

// device arrays of n values
extern "C" int table_entries() { return CIS_N; }
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


def both_signs(x):
    return np.concatenate([x, -x])


def test_rsqrt64(lib):
    """The estimate's relative error 2^-22 cubed is far below the rounding of the step: the residual's error counts half,
    the last addition rounds once: 1.5 units of 2^-53 and the unit's change at a power of two, 3 units."""
    rng = np.random.default_rng(1)
    x = np.concatenate([rng.uniform(1, 4, 200_000), 2.0 ** rng.uniform(-300, 300, 200_000), 4.0 ** np.arange(-150, 150),
                        np.nextafter(4.0 ** np.arange(-150, 150), 0), np.nextafter(4.0 ** np.arange(-150, 150), np.inf)])
    exact = 1 / np.sqrt(x.astype(np.longdouble))
    assert np.abs(evaluate(lib, 1, 1, x)[0] / exact - 1).max() <= 3 * 2.0 ** -53


def test_rcp64(lib):
    """As rsqrt64: 3 units of 2^-53."""
    rng = np.random.default_rng(2)
    x = both_signs(np.concatenate([rng.uniform(1, 2, 200_000), 2.0 ** rng.uniform(-300, 300, 200_000),
                                   2.0 ** np.arange(-300, 300), np.nextafter(2.0 ** np.arange(-300, 300), 0)]))
    assert np.abs(evaluate(lib, 2, 1, x)[0] * x.astype(np.longdouble) - 1).max() <= 3 * 2.0 ** -53


@pytest.mark.parametrize("kappa", [0.0, 0.37, 5.0, 27.0, 1000.0])
def test_phase64(lib, kappa):
    """exp(i kappa r), r from 1e-9 to 100, with the midpoints and the entries of the table: the entry rounds once, the
    product three times (0.5 and 1.5 units of 2^-53), the argument's remainder within half an entry (pi / 1024) to 2^-53 of
    itself: 2.5 units."""
    n = lib.table_entries()
    k = np.arange(n)
    angle = 8 * np.arctan(np.longdouble(1)) * k / n
    tab = np.cos(angle).astype(float) + 1j * np.sin(angle).astype(float)
    rng = np.random.default_rng(3)
    r = np.concatenate([rng.uniform(0, 5, 200_000), 10.0 ** rng.uniform(-9, 2, 100_000), (k + 0.5) * np.pi * 2 / n, k * np.pi * 2 / n])
    got = evaluate(lib, 3, 2, np.full(r.size, kappa), r, np.pad(tab.view(np.float64), (0, max(0, r.size - 2 * n))))
    phase = np.longdouble(kappa) * r.astype(np.longdouble)
    tol = 2.5 * 2.0 ** -53 + phase * np.finfo(np.longdouble).eps  # the host's product rounds too
    assert (np.abs(got[0] - np.cos(phase)) <= tol).all() and (np.abs(got[1] - np.sin(phase)) <= tol).all()


def test_sin_cosm1(lib):
    """Up to 1e6, all quadrants: the reduction rounds twice at pi / 4 (2^-24 each at most), the series and the last sum about as
    much, 4 x 2^-24 together; below pi / 4, relative to the values: 3 roundings and the term left out, 4 x 2^-24."""
    rng = np.random.default_rng(4)
    x = np.float32(both_signs(np.concatenate([rng.uniform(0, 20, 200_000), 10.0 ** rng.uniform(0, 6, 200_000),
                                              np.arange(1, 2000) * np.pi / 4]))).astype(float)
    s, c = evaluate(lib, 4, 2, x)
    assert np.abs(s - np.sin(x)).max() <= 4 * 2.0 ** -24 and np.abs(c + 1 - np.cos(x)).max() <= 4 * 2.0 ** -24
    x = np.float32(both_signs(10.0 ** rng.uniform(-15, np.log10(0.785), 200_000))).astype(float)
    s, c = evaluate(lib, 4, 2, x)
    assert np.abs(s / np.sin(x) - 1).max() <= 4 * 2.0 ** -24
    assert np.abs(c / (-2 * np.sin(x / 2) ** 2) - 1).max() <= 4 * 2.0 ** -24


def test_two_sum(lib):
    """Sum and rounding errors together are exact while the errors themselves fit in FP32 (here three values within 2^20 of
    one another: the errors of two additions, 2^-24 and below, add without rounding to 2^-47)."""
    rng = np.random.default_rng(5)
    v = [np.float32(rng.standard_normal(100_000) * 2.0 ** rng.uniform(-10, 10, 100_000)).astype(float) for _ in range(3)]
    got = evaluate(lib, 5, 1, *v)[0]
    assert np.abs(got - (v[0] + v[1] + v[2])).max() <= 2.0 ** -47 * np.abs(v).sum(axis=0).max()

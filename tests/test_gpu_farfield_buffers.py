"""Where igabem_farfield puts its result: device memory at an 8-byte boundary (complex doubles that a caller's own
layout does not align to 16 bytes), which the kernels' 16-byte stores cannot write in place, equals the same
call's result in aligned device memory and in host memory.

Tolerance: FP64 runs the same operations in the same order, equal bits; FP32 adds its groups by atomics, so runs
differ by a few roundings of the FP64 sums: 1e-14."""
import numpy as np
import pytest

from paper_2306_11324_gb300 import binding as B
from paper_2306_11324_gb300 import inputs
from tests import gpu_util as G

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", [B.FP64, B.MIXED_FP32])
@pytest.mark.parametrize("n_dir,columns", [(1, 1), (37, 3), (130, 5)])
def test_result_at_an_8_byte_boundary(precision, n_dir, columns):
    import torch
    prob, info = G.problem(level_m=1, degree_p=1, kappa=2.0, eta_cfie=1.0, no_fmm=1, precision=precision)
    x = torch.from_numpy(inputs.random_complex(info["n_dofs"], seed=n_dir, cols=columns)).cuda()
    xh = inputs.fibonacci_directions(n_dir)
    aligned = B.igabem_farfield(prob, x, xh).cpu().numpy()
    host = B.igabem_farfield(prob, x, xh, np.empty((n_dir, columns), np.complex128))
    buf = torch.full((2 + 2 * n_dir * columns,), np.nan, dtype=torch.float64, device="cuda")
    odd = buf[1:-1]
    assert odd.data_ptr() % 16 == 8
    B.igabem_farfield(prob, x, xh, odd)
    got = odd.cpu().numpy().view(np.complex128).reshape(n_dir, columns)
    tol = 0.0 if precision == B.FP64 else 1e-14
    assert G.rel(got, aligned) <= tol and G.rel(host, aligned) <= tol
    assert torch.isnan(buf[0]) and torch.isnan(buf[-1])
    B.igabem_problem_destroy(prob)

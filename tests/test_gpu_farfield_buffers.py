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


def test_memory_of_the_call_is_counted_and_given_back():
    """The problem's device_bytes follow the buffer it keeps, and a call of 88 MB leaves no more than that behind (to the
    2 MB of cudaMalloc's granularity on either side)."""
    import torch
    prob, info = G.problem(level_m=1, degree_p=1, kappa=2.0, eta_cfie=1.0, no_fmm=1)
    x = inputs.random_complex(info["n_dofs"], seed=1, cols=4)
    B.igabem_farfield(prob, x, inputs.fibonacci_directions(40))    # work buffers and kernels are there
    held = B.igabem_problem_info(prob)["device_bytes"]
    free = torch.cuda.mem_get_info()[0]
    for n_dir in (200_000, 1_000_000, 40):
        B.igabem_farfield(prob, x, inputs.fibonacci_directions(n_dir))
        more = B.igabem_problem_info(prob)["device_bytes"] - held
        assert free - torch.cuda.mem_get_info()[0] <= more + (4 << 20)
        assert more <= 32 << 20
    B.igabem_problem_destroy(prob)

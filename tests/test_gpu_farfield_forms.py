"""The FP32 far-field kernel's forms (one, two and four directions a thread, by the blocks that fill the device) against
the FP64 one: direction counts that end a form's blocks early, columns around its passes of 8, both boundary
conditions.

Tolerance (max-norm relative): FP32 phases of a group of elements and sums of its points, about 50 eps: 4e-6."""
import numpy as np
import pytest

from paper_2306_11324_gb300 import binding as B
from paper_2306_11324_gb300 import inputs
from tests import gpu_util as G

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("hard", [False, True])
@pytest.mark.parametrize("n_dir,columns", [(1, 3), (2900, 9), (5901, 3), (6144, 8), (20001, 9), (30000, 1)])
def test_fp32_far_field_equals_fp64(hard, n_dir, columns):
    u = []
    for precision in (B.FP64, B.MIXED_FP32):
        prob, info = G.problem(level_m=2, degree_p=2, kappa=6.0, eta_cfie=1.0, bc=int(hard), cheb_q=3, leaf_offset=1,
                               precision=precision)
        x = inputs.random_complex(info["n_dofs"], seed=n_dir, cols=columns)
        u.append(B.igabem_farfield(prob, x, inputs.fibonacci_directions(n_dir)))
        B.igabem_problem_destroy(prob)
    assert np.isfinite(u[1]).all() and G.rel(u[1], u[0]) < 4e-6


@pytest.mark.parametrize("hard", [False, True])
@pytest.mark.parametrize("n_dir", [1, 200, 700])
def test_fp64_column_alone_equals_columns_together(hard, n_dir):
    """The single column's kernel and the four columns' one add the same terms in the same order; the compiler may contract
    them differently: 1e-13."""
    prob, info = G.problem(level_m=3, degree_p=2, kappa=6.0, eta_cfie=1.0, bc=int(hard), cheb_q=3, leaf_offset=1)
    x = inputs.random_complex(info["n_dofs"], seed=n_dir, cols=3)
    xh = inputs.fibonacci_directions(max(n_dir, 2))[:n_dir]
    together = B.igabem_farfield(prob, x, xh)
    for r in range(3):
        assert G.rel(B.igabem_farfield(prob, np.ascontiguousarray(x[:, r:r + 1]), xh), together[:, r:r + 1]) < 1e-13
    B.igabem_problem_destroy(prob)

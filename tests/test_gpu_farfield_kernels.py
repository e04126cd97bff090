"""The far-field kernels against the defining sum in 64-bit numpy (oracle): direction counts around the FP32 kernel's
blocks (1, 64, 65, 128, 129, 300) and the FP64 kernel's clusters, column counts around its passes of 8 (FP32) and
4 (FP64), both boundary conditions.

Tolerances (max-norm relative): FP64 1e-10, the suite's bound; FP32 phases of a group of 16 x 16 elements and sums of
its points, about 50 eps: 4e-6, below the 1e-5 the mixed precision is held to."""
import numpy as np
import pytest

from oracle import farfield
from paper_2306_11324_gb300 import binding as B
from paper_2306_11324_gb300 import inputs
from tests import gpu_util as G
from tests import oracle_cache as C

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("hard", [False, True])
@pytest.mark.parametrize("precision,tol", [(B.FP64, 1e-10), (B.MIXED_FP32, 4e-6)])
@pytest.mark.parametrize("n_dir,columns", [(1, 1), (64, 3), (65, 4), (128, 5), (129, 8), (300, 9), (700, 2)])
def test_far_field(hard, precision, tol, n_dir, columns):
    prob, info = G.problem(level_m=2, degree_p=2, kappa=6.0, eta_cfie=1.0, bc=int(hard), cheb_q=3, leaf_offset=1,
                           precision=precision)
    sp = C.sphere_space(2, 2, hard)
    x = inputs.random_complex(sp.N, seed=n_dir, cols=columns)
    xh = inputs.fibonacci_directions(n_dir)
    ref = np.stack([farfield.far_field(sp, 6.0, x[:, r], xh, hard) for r in range(columns)], axis=1)
    assert G.rel(B.igabem_farfield(prob, x, xh), ref) < tol
    B.igabem_problem_destroy(prob)

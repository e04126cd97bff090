"""On-the-fly M2L of sound-hard problems in the mixed precision with 24 to 47 columns, on both sides of the rule between
its two kernels (column count, q, clusters): the product with all columns against the same columns five at a time.

Tolerance (max-norm relative): FP32 sums in another order, the mixed product's bound, 2e-6."""
import numpy as np
import pytest

from paper_2306_11324_gb300 import binding as B
from paper_2306_11324_gb300 import inputs

from .gpu_util import problem, rel

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m,q", [(3, 5), (3, 8), (4, 4), (4, 7)])
def test_columns_together_equal_columns_apart(m, q):
    prob, info = problem("deformed", level_m=m, degree_p=2, kappa=4.0, eta_cfie=0.6, bc=1, cheb_q=q, leaf_offset=1,
                         precision=B.MIXED_FP32)
    x = inputs.random_complex(info["n_dofs"], seed=m, cols=47)
    apart = np.concatenate([B.igabem_matvec(prob, np.ascontiguousarray(x[:, r:r + 5])) for r in range(0, 47, 5)], axis=1)
    for R in (24, 27, 28, 35, 36, 47):
        assert rel(B.igabem_matvec(prob, np.ascontiguousarray(x[:, :R])), apart[:, :R]) < 2e-6
    B.igabem_problem_destroy(prob)

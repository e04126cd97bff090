"""Products with stored blocks (k_stream): the near field and the stored M2L against the same operator's columns
taken one at a time and against the on-the-fly M2L, at block sizes with one or many pairs side by side in a
thread block (rows 4 .. 256), column counts around the kernel's widths (1, 2, 4, 6, 8, 10, 12, 16 and several
passes, odd and even), both precisions and boundary conditions, split and unsplit lists.

Tolerances (max-norm relative): FP64 sums of a few thousand terms differ by their order alone: 1e-13.  FP32: the
block's sums in another order, about 20 eps: 2e-6, the mixed product's bound."""
import numpy as np
import pytest

from paper_2306_11324_gb300 import binding as B
from paper_2306_11324_gb300 import inputs

from .gpu_util import problem, rel

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("hard", [False, True])
@pytest.mark.parametrize("precision,tol", [(B.FP64, 1e-13), (B.MIXED_FP32, 2e-6)])
@pytest.mark.parametrize("m,p,b,q,stored", [(2, 1, 0, 3, 1), (3, 1, 1, 4, 1), (3, 2, 1, 7, 1), (3, 3, 1, 12, 1),
                                            (4, 2, 2, 7, 1), (4, 1, 3, 9, 0), (4, 2, 2, 7, 0)])
def test_columns_together_equal_columns_alone(hard, precision, tol, m, p, b, q, stored):
    prob, info = problem("deformed", level_m=m, degree_p=p, kappa=4.0, eta_cfie=0.6, bc=int(hard), cheb_q=q,
                         leaf_offset=b, precision=precision, m2l_stored=stored)
    N = info["n_dofs"]
    x = inputs.random_complex(N, seed=m, cols=33)
    one = np.concatenate([B.igabem_matvec(prob, np.ascontiguousarray(x[:, r:r + 1])) for r in range(33)], axis=1)
    for R in (2, 3, 5, 6, 9, 11, 16, 17, 33):
        y = B.igabem_matvec(prob, np.ascontiguousarray(x[:, :R]))
        assert rel(y, one[:, :R]) < tol
    B.igabem_problem_destroy(prob)

"""Moments and fields of the band levels (k_p2m_band, k_l2p_band): a cluster's rows of Gauss points split over thread
blocks (few columns: clusters of up to 8) against the same rows in one block (many columns), both precisions and
boundary conditions.

Tolerances (max-norm relative): FP64 sums of a few thousand terms differ by their order alone: 1e-13.  FP32: the sums
in another order, the mixed product's bound, 2e-6."""
import numpy as np
import pytest

from paper_2306_11324_gb300 import binding as B
from paper_2306_11324_gb300 import inputs

from .gpu_util import problem, rel

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("hard", [False, True])
@pytest.mark.parametrize("precision,tol", [(B.FP64, 1e-13), (B.MIXED_FP32, 2e-6)])
@pytest.mark.parametrize("m,p,b,q,q_max,cap", [(4, 1, 1, 4, 10, 2.0), (5, 2, 2, 6, 9, 4.0)])
def test_columns_alone_equal_columns_together(hard, precision, tol, m, p, b, q, q_max, cap):
    prob, info = problem("deformed", level_m=m, degree_p=p, kappa=16.0, eta_cfie=0.6, bc=int(hard), cheb_q=q,
                         q_max=q_max, kappa_cap=cap, leaf_offset=b, precision=precision)
    assert len(set(info["level_q"][:info["n_levels"]])) > 1  # the levels differ, so there are bands
    R = 160 if m < 5 else 40
    x = inputs.random_complex(info["n_dofs"], seed=m, cols=R)
    y = B.igabem_matvec(prob, x)
    for r in (0, R - 1):
        assert rel(B.igabem_matvec(prob, np.ascontiguousarray(x[:, r:r + 1])), y[:, r:r + 1]) < tol
    assert rel(B.igabem_matvec(prob, np.ascontiguousarray(x[:, 3:10])), y[:, 3:10]) < tol
    B.igabem_problem_destroy(prob)

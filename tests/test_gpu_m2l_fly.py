"""On-the-fly M2L (k_m2l_fly, k_m2l_gemm) against the stored coupling blocks of the same operator, whose
samples come from CUDA's sincos and rsqrt: every q whose block layout differs (one or several pairs side
by side in a block, one pair per block), column counts on both sides of the kernel's widths, both boundary
conditions, split and unsplit interaction lists.

Tolerances (max-norm relative, FP64): each side's samples carry a few roundings of the phase kappa r <= 20 and
of 1/r (about 20 eps = 4e-15 together) and sums of up to 200 q^2 terms add about as much: 1e-13.  FP32: the
same roundings at 6e-8 with the phase split (no growth with kappa r): 2e-6, the mixed product's bound."""
import numpy as np
import pytest

from paper_2306_11324_gb300 import binding as B
from paper_2306_11324_gb300 import inputs

from .gpu_util import problem, rel

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("hard", [False, True])
@pytest.mark.parametrize("precision,tol", [(B.FP64, 1e-13), (B.MIXED_FP32, 2e-6)])
@pytest.mark.parametrize("q,m,b,columns", [(2, 3, 1, (1, 5)), (5, 3, 1, (2, 3)), (7, 3, 1, (1, 3, 4, 7, 26)),
                                           (8, 3, 1, (1, 25, 48)), (11, 3, 1, (1, 6)), (12, 3, 1, (3,)),
                                           (16, 2, 0, (1, 2)), (7, 5, 2, (1, 4))])
def test_on_the_fly_equals_stored_blocks(hard, precision, tol, q, m, b, columns):
    kw = dict(level_m=m, degree_p=1 if b == 0 else 2, kappa=5.0, eta_cfie=0.7, bc=int(hard), cheb_q=q, leaf_offset=b,
              precision=precision)
    fly, info = problem("deformed" if m >= 2 else "sphere", **kw)
    stored, _ = problem("deformed" if m >= 2 else "sphere", m2l_stored=1, **kw)
    assert info["n_far_pairs"] > 0
    for R in columns:
        x = inputs.random_complex(info["n_dofs"], seed=R, cols=R)
        assert rel(B.igabem_matvec(fly, x), B.igabem_matvec(stored, x)) < tol
    B.igabem_problem_destroy(fly)
    B.igabem_problem_destroy(stored)

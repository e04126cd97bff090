"""One operator with leaves of every size: with every pair in the near field (a tiny eta_adm) the leaf size decides the
blocks' rows, the kernel that fills them (leaf pairs as a whole for leaves of up to 4 x 4 elements and p <= 2, element
pairs otherwise) and the kernel that multiplies them (k_stream up to 256 rows, k_near_spmv2 above), and the product must
not depend on it.  Rows per block 4 .. 289.

Tolerances (max-norm relative): FP64 sums in another order, samples by the table-driven phase on one side and CUDA's sincos
on the other, 1e-12; FP32 samples and sums against FP64, the mixed product's bound, 2e-6."""
import numpy as np
import pytest

from paper_2306_11324_gb300 import binding as B
from paper_2306_11324_gb300 import inputs

from .gpu_util import problem, rel

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m,p,leaves,hard", [(4, 1, (3, 4), False), (3, 2, (0, 2, 3), False), (3, 4, (2, 3), False),
                                             (3, 6, (1, 3), False), (4, 1, (3, 4), True), (3, 2, (0, 2, 3), True),
                                             (3, 4, (2, 3), True)])
def test_leaf_size_does_not_matter(m, p, leaves, hard):
    kw = dict(level_m=m, degree_p=p, kappa=3.0, eta_cfie=0.7, bc=int(hard), cheb_q=4, eta_adm=1e-6)
    ref, info = problem("deformed", leaf_offset=1 if p < 6 else 2, **kw)
    assert info["n_far_pairs"] == 0
    x = inputs.random_complex(info["n_dofs"], seed=m, cols=17)
    y = np.concatenate([B.igabem_matvec(ref, np.ascontiguousarray(x[:, r:r + 1])) for r in range(17)], axis=1)
    B.igabem_problem_destroy(ref)
    for b in leaves:
        for precision, tol in ((B.FP64, 1e-12), (B.MIXED_FP32, 2e-6)):
            prob, _ = problem("deformed", leaf_offset=b, precision=precision, **kw)
            for R in (1, 3, 17):
                assert rel(B.igabem_matvec(prob, np.ascontiguousarray(x[:, :R])), y[:, :R]) < tol, (b, precision, R)
            B.igabem_problem_destroy(prob)


@pytest.mark.parametrize("R", [208, 256, 400, 512])
def test_tensor_core_slices(R):
    """Sound-soft widths with two slices in a group (208 to 256 columns) and with three groups (400 to 512): the
    columns together and sixteen at a time, FP32 sums in another order, 2e-6."""
    prob, info = problem("deformed", level_m=3, degree_p=2, kappa=4.0, eta_cfie=0.7, cheb_q=7, leaf_offset=1,
                         precision=B.MIXED_TC)
    x = inputs.random_complex(info["n_dofs"], seed=R, cols=R)
    y = B.igabem_matvec(prob, x)
    for r in range(0, R, 16 if R < 300 else 80):
        assert rel(y[:, r:r + 16], B.igabem_matvec(prob, np.ascontiguousarray(x[:, r:r + 16]))) < 2e-6
    B.igabem_problem_destroy(prob)

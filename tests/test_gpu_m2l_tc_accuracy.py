"""Rounding of the tensor-core M2L: rows of a product that only far couplings reach (the density on one patch of the
deformed sphere, the rows of the patch opposite to it) against the FP64 product.

Tolerance (root mean square, relative).  An instruction truncates the FP32 sum it adds to, half a unit in the last
place on average, 2^-24 of the sum so far.  With the small products first, the 7 instructions of the last
third see the sum grow from nothing to the whole: 3.5 x 2^-24 = 2.1e-7.  The FP32 samples, phases and sums add what the
FP32 M2L shows on these rows, at most 2.5e-7: together 3.3e-7 by squares, and a fifth more for what the estimate
leaves out: 4e-7.  (Products in any order of K alone: 14 to 21 instructions at half to all of the sum, 4.8e-7 to
7.5e-7 measured.)"""
import numpy as np
import pytest

from paper_2306_11324_gb300 import binding as B
from paper_2306_11324_gb300 import inputs

from .gpu_util import problem

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m,kappa,columns,coherent", [(3, 0.0, 16, True), (3, 5.0, 16, False), (4, 11.0, 16, True),
                                                      (4, 11.0, 64, False), (4, 11.0, 208, False)])
def test_far_rows_against_fp64(m, kappa, columns, coherent):
    centre = [np.asarray(p.ctrl).reshape(-1, 3).mean(axis=0) for p in inputs.deformed_sphere_patches(spans=4)]
    opposite = int(np.argmin([c @ centre[0] for c in centre]))
    nb = (2 ** m + 2) ** 2  # unknowns of a patch
    y = {}
    for precision in (B.FP64, B.MIXED_TC):
        prob, info = problem("deformed", level_m=m, degree_p=2, kappa=kappa, eta_cfie=1.0, cheb_q=7, leaf_offset=1,
                             precision=precision)
        x = np.zeros((info["n_dofs"], columns), complex)
        x[:nb] = 1.0 if coherent else inputs.random_complex(info["n_dofs"], seed=3, cols=columns)[:nb]
        y[precision] = B.igabem_matvec(prob, x)[opposite * nb:(opposite + 1) * nb]
        B.igabem_problem_destroy(prob)
    assert np.linalg.norm(y[B.MIXED_TC] - y[B.FP64]) < 4e-7 * np.linalg.norm(y[B.FP64])

"""Rounding of the FP32 M2L on the fly: rows of a product that only far couplings reach (random densities on one patch
of the deformed sphere, the rows of the patch opposite to it) against the FP64 product, at the largest q.

Tolerance (root mean square, relative).  Summing the q^2 = 256 products of a pair in one chain rounds to about
sqrt(256 / 2) = 11 units of 2.5e-8 of the pair's sum, in blocks of q to sqrt(16 / 2 + 16 / 2) = 4; the transfers behind
it average over the nodes.  Measured on these rows with blocks of q 5.0e-8 to 5.2e-8, with one chain 6.5e-8 to 6.8e-8; the
bound lies half way, 5.8e-8.  (With 16 columns the moments' form for many columns adds 1.9e-7 here, either way.)"""
import numpy as np
import pytest

from paper_2306_11324_gb300 import binding as B
from paper_2306_11324_gb300 import inputs

from .gpu_util import problem

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("columns", [1, 4])
def test_far_rows_against_fp64(columns):
    centre = [np.asarray(p.ctrl).reshape(-1, 3).mean(axis=0) for p in inputs.deformed_sphere_patches(spans=4)]
    opposite = int(np.argmin([c @ centre[0] for c in centre]))
    nb, y = 10 * 10, {}  # unknowns of a patch
    for precision in (B.FP64, B.MIXED_FP32):
        prob, info = problem("deformed", level_m=3, degree_p=2, kappa=0.0, eta_cfie=1.0, cheb_q=16, leaf_offset=1,
                             precision=precision)
        x = np.zeros((info["n_dofs"], columns), complex)
        x[:nb] = inputs.random_complex(info["n_dofs"], seed=3, cols=columns)[:nb]
        y[precision] = B.igabem_matvec(prob, x)[opposite * nb:(opposite + 1) * nb]
        B.igabem_problem_destroy(prob)
    assert np.linalg.norm(y[B.MIXED_FP32] - y[B.FP64]) < 5.8e-8 * np.linalg.norm(y[B.FP64])

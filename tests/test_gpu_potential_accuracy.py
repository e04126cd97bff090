"""Rounding of the potential's octree in the mixed precision (k_pot_m2l<float>) against the FP64 form with the same
interpolation, at wavenumbers from a static field to a dozen wavelengths, and its range of densities.

Tolerances (root mean square, relative).  A sample, an expansion and the sum of 16 products round to about 8e-8 of the
part of the kernel that is formed in FP32, 343 of them add up like a random walk.  Where the phase hardly turns
within a box that part is a fifth of the kernel: sound-soft, monopoles, 8e-8 / 5 / sqrt(343) = 1e-9, bound 1e-8; sound-hard, the
moments of a box cancel, and an FP32 kernel of full size shows 1.3e-6 of the field with 5e-8 a sample: 1.3e-6 x 8 / 5 / 5 =
4e-7, bound 6e-7.  With more phase the part grows to the kernel itself: 5e-8 a sample and the phase's 6e-8 kappa r give
1.5e-7 at kappa = 12, bound 3e-7."""
import numpy as np
import pytest

from paper_2306_11324_gb300 import binding as B
from paper_2306_11324_gb300 import inputs

from .gpu_util import problem

pytestmark = pytest.mark.gpu


def points(n):
    rng = np.random.default_rng(n)
    p = rng.standard_normal((n, 3))
    return p * rng.uniform(1.6, 4.0, (n, 1)) / np.linalg.norm(p, axis=1, keepdims=True)


@pytest.mark.parametrize("kappa,hard,tol", [(0.0, False, 1e-8), (0.3, False, 1e-8), (0.5, True, 6e-7), (3.0, False, 3e-7),
                                            (3.0, True, 6e-7), (12.0, False, 3e-7)])
def test_fp32_tree_against_fp64(kappa, hard, tol):
    u = {}
    for precision in (B.FP64, B.MIXED_FP32):
        prob, info = problem("deformed", level_m=3, degree_p=2, kappa=kappa, eta_cfie=0.7, bc=int(hard), cheb_q=7,
                             leaf_offset=2, precision=precision)
        u[precision] = B.igabem_potential(prob, inputs.random_complex(info["n_dofs"], seed=3, cols=1), points(2000))
        B.igabem_problem_destroy(prob)
    assert np.linalg.norm(u[B.MIXED_FP32] - u[B.FP64]) < tol * np.linalg.norm(u[B.FP64])


@pytest.mark.parametrize("exponent", [-900, -160, 160, 900])
def test_densities_beyond_the_range_of_fp32(exponent):
    """The field is linear in the density: scaled by a power of two, the same bits scaled."""
    prob, info = problem("deformed", level_m=2, degree_p=1, kappa=2.0, eta_cfie=0.7, cheb_q=5, leaf_offset=1,
                         precision=B.MIXED_FP32)
    x = inputs.random_complex(info["n_dofs"], seed=3, cols=2)
    u = B.igabem_potential(prob, x, points(300))
    assert np.array_equal(B.igabem_potential(prob, x * 2.0 ** exponent, points(300)), u * 2.0 ** exponent)
    B.igabem_problem_destroy(prob)

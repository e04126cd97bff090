"""The potential's interaction lists where only the finest boxes are admissible (a small phase cap): box offsets up to the
whole cube, which are sorted instead of counted, against the direct sum.

Tolerance (max-norm relative): q = 6 nodes over boxes at half their distance with a phase of 0.1, the interpolation error of
1 / r: 1e-4."""
import numpy as np
import pytest

from paper_2306_11324_gb300 import binding as B
from paper_2306_11324_gb300 import inputs

from .gpu_util import problem, rel

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("cap", [0.1, 6.0])
def test_lists_of_the_finest_level(cap):
    kw = dict(level_m=4, degree_p=1, kappa=1.0, eta_cfie=1.0, cheb_q=6, leaf_offset=2, precision=B.MIXED_FP32)
    tree, info = problem("sphere", kappa_cap=cap, **kw)
    direct, _ = problem("sphere", no_fmm=1, leaf_offset=4, **{k: v for k, v in kw.items() if k != "leaf_offset"})
    rng = np.random.default_rng(1)
    pts = rng.standard_normal((1500, 3))
    pts *= rng.uniform(1.3, 4.0, (1500, 1)) / np.linalg.norm(pts, axis=1, keepdims=True)
    x = np.ones((info["n_dofs"], 1), complex) + inputs.random_complex(info["n_dofs"], seed=1, cols=1)
    assert rel(B.igabem_potential(tree, x, pts), B.igabem_potential(direct, x, pts)) < 1e-4
    B.igabem_problem_destroy(tree)
    B.igabem_problem_destroy(direct)

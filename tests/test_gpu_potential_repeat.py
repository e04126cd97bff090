"""igabem_potential on the same inputs gives the same bits: every sum has a fixed order, on levels whose pairs fill the
result buffer several times (the last case: 8 densities, 44 MB a thousand pairs) as on small ones."""
import numpy as np
import pytest

from paper_2306_11324_gb300 import binding as B
from paper_2306_11324_gb300 import inputs

from .gpu_util import problem

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", [B.FP64, B.MIXED_FP32])
@pytest.mark.parametrize("m,q,hard,columns,points", [(2, 5, False, 1, 700), (2, 4, True, 3, 500), (3, 7, False, 8, 1500)])
def test_calls_repeat_bit_for_bit(precision, m, q, hard, columns, points):
    prob, info = problem("deformed", level_m=m, degree_p=2, kappa=3.0, eta_cfie=0.7, bc=int(hard), cheb_q=q, leaf_offset=1,
                         precision=precision)
    rng = np.random.default_rng(points)
    pts = rng.standard_normal((points, 3))
    pts *= rng.uniform(1.6, 4.0, (points, 1)) / np.linalg.norm(pts, axis=1, keepdims=True)
    x = inputs.random_complex(info["n_dofs"], seed=m, cols=columns)
    first = B.igabem_potential(prob, x, pts)
    assert np.isfinite(first).all()
    for _ in range(3):
        assert np.array_equal(B.igabem_potential(prob, x, pts), first)
    B.igabem_problem_destroy(prob)

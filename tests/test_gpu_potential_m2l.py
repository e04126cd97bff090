"""The octree's M2L by box offsets (k_pot_m2l): FP32 against FP64 samples of the same interpolated kernel, at
node counts with partial row blocks (q^3 below, at and above 128 rows and 64 source nodes), column counts
that fill, underfill and split a chunk of 16, and both representations.

Tolerance (max-norm relative): the FP32 samples and sums carry a few FP32 roundings each, the phase split
keeps them from growing with kappa r: 2e-6, the mixed precision's bound for one product."""
import numpy as np
import pytest

from paper_2306_11324_gb300 import binding as B
from paper_2306_11324_gb300 import inputs

from .gpu_util import problem, rel

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("hard", [False, True])
@pytest.mark.parametrize("q,columns", [(2, 1), (4, 3), (5, 8), (7, 1), (7, 5), (8, 2), (10, 1)])
def test_fp32_tree_equals_fp64_tree(hard, q, columns):
    kw = dict(level_m=2, degree_p=2, kappa=2.5, eta_cfie=1.0, bc=int(hard), cheb_q=q, leaf_offset=1)
    p64, info = problem("sphere", **kw)
    p32, _ = problem("sphere", precision=B.MIXED_FP32, **kw)
    rng = np.random.default_rng(q)
    # clusters of points (boxes with many targets) and single points far out
    pts = np.concatenate([inputs.fibonacci_directions(40) * r for r in (1.5, 3.0, 9.0)] +
                         [np.array([0.0, 0.0, 5.0]) + 0.2 * rng.standard_normal((300, 3))])
    x = inputs.random_complex(info["n_dofs"], seed=columns, cols=columns)
    assert rel(B.igabem_potential(p32, x, pts), B.igabem_potential(p64, x, pts)) < 2e-6
    B.igabem_problem_destroy(p64)
    B.igabem_problem_destroy(p32)

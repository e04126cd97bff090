"""GMRES with as many columns as the server merges (the Arnoldi kernel takes four columns a block, the last block to
finish advances the iteration): columns that finish at different iterations, several cycles, a second solve on the same
buffers with fewer columns, against LU on a dense system.

Tolerance: GMRES stops at a relative residual of 1e-10; the condition number of these systems is below 100."""
import numpy as np
import pytest

from oracle import assemble as A
from oracle import solve
from paper_2306_11324_gb300 import binding as B
from paper_2306_11324_gb300 import inputs
from tests import gpu_util as G
from tests import oracle_cache as C

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("restart", [9, 40])
def test_wide_solves_match_lu(restart):
    prob, info = G.problem(level_m=2, degree_p=1, kappa=2.0, eta_cfie=0.5, bc=1, no_fmm=1, tol=1e-10, max_iter=2000,
                           gmres_restart=restart)
    sp = C.sphere_space(2, 1, True)
    Amat = C.cfie(2, 1, 2.0, 0.5, True)
    for columns in (256, 67, 4):
        d = inputs.fibonacci_directions(columns)
        x, s = B.igabem_solve(prob, d, info["n_dofs"])
        ref = solve.lu_solve(Amat, np.stack([A.rhs(sp, 2.0, 0.5, v, True) for v in d], axis=1))
        assert s["rel_residual"] <= 1e-10
        assert G.rel(x, ref) < 1e-8
    B.igabem_problem_destroy(prob)

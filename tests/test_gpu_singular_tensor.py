"""Touching pairs in tensor form (k_sing_tensor) against the oracle's rules, entry by entry through the dense operator
(no_fmm): every degree it takes, both boundary conditions, geometry degrees 2 and 4, and meshes whose
touching pairs meet across patches in every relative position.

Tolerance (max-norm relative, FP64): the suite's bound for the dense matrix, 1e-10; the two forms add the same
125-point slabs in another order, a few hundred roundings."""
import numpy as np
import pytest

from oracle import assemble as A
from oracle import space as S
from paper_2306_11324_gb300 import binding as B
from paper_2306_11324_gb300 import inputs
from tests import gpu_util as G

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("hard,p", [(False, 0), (False, 1), (False, 2), (False, 3), (True, 1), (True, 2), (True, 3)])
@pytest.mark.parametrize("kind", ["sphere", "torus"])
def test_operator_matches_oracle(kind, hard, p):
    patches = inputs.unit_sphere_patches() if kind == "sphere" else inputs.torus_patches()
    m, kappa, eta = 1, 1.3, 0.8
    geom = B.igabem_geometry_create(G.ctx(), patches)
    prob = B.igabem_problem_create(geom, B.igabem_default_options(level_m=m, degree_p=p, kappa=kappa, eta_cfie=eta,
                                                                  bc=int(hard), no_fmm=1))
    sp = S.Space(S.Mesh(patches, m), p, continuous=hard)
    x = inputs.random_complex(sp.N, seed=5, cols=2)
    ref = A.cfie_matrix(sp, kappa, eta, hard) @ x
    assert G.rel(B.igabem_matvec(prob, x), ref) < 1e-10
    B.igabem_problem_destroy(prob)
    B.igabem_geometry_destroy(geom)

"""Regular pairs of a sound-soft near field, leaf pair by leaf pair (k_near_tensor), against the oracle's rules entry by
entry through the dense operator (no_fmm: one leaf per patch): every degree it takes, leaves of 1, 2 and 4 elements
per direction (16, 4 and 1 leaf pairs in a thread block, the last block partly filled), both precisions, leaf pairs
that touch along an edge, at a corner or not at all.

Tolerances (max-norm relative): FP64, the suite's bound for the dense matrix, 1e-10; FP32 samples and sums, the mixed
product's bound, 2e-6."""
from functools import lru_cache

import pytest

from oracle import assemble as A
from oracle import space as S
from paper_2306_11324_gb300 import binding as B
from paper_2306_11324_gb300 import inputs
from tests import gpu_util as G

pytestmark = pytest.mark.gpu
KAPPA, ETA = 1.3, 0.8


@lru_cache(maxsize=None)
def reference(kind, m, p):
    patches = inputs.unit_sphere_patches() if kind == "sphere" else inputs.torus_patches()
    sp = S.Space(S.Mesh(patches, m), p, continuous=False)
    x = inputs.random_complex(sp.N, seed=5, cols=2)
    return patches, x, A.cfie_matrix(sp, KAPPA, ETA, False) @ x


@pytest.mark.parametrize("precision,tol", [(B.FP64, 1e-10), (B.MIXED_FP32, 2e-6)])
@pytest.mark.parametrize("p", [0, 1, 2])
@pytest.mark.parametrize("kind,m", [("sphere", 0), ("sphere", 1), ("sphere", 2), ("torus", 0)])
def test_operator_matches_oracle(kind, m, p, precision, tol):
    patches, x, ref = reference(kind, m, p)
    geom = B.igabem_geometry_create(G.ctx(), patches)
    prob = B.igabem_problem_create(geom, B.igabem_default_options(level_m=m, degree_p=p, kappa=KAPPA, eta_cfie=ETA,
                                                                  bc=0, no_fmm=1, precision=precision))
    assert G.rel(B.igabem_matvec(prob, x), ref) < tol
    B.igabem_problem_destroy(prob)
    B.igabem_geometry_destroy(geom)

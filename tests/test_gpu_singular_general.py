"""The general singular kernel (k_near_singular), which takes degrees above 3 and singular rules of other than five
points, and the sound-hard regular pairs of both precisions (k_near_tensor in FP32, k_near_regular_f in FP64), against
the oracle's rules entry by entry through the dense operator (no_fmm).

Tolerances (max-norm relative): FP64, the suite's bound for the dense matrix, 1e-10; FP32 regular pairs, the mixed
product's bound, 2e-6."""
import functools

import pytest

from oracle import assemble as A
from oracle import space as S
from paper_2306_11324_gb300 import binding as B
from paper_2306_11324_gb300 import inputs
from tests import gpu_util as G

pytestmark = pytest.mark.gpu
KAPPA, ETA = 1.3, 0.8


@functools.lru_cache(maxsize=None)
def reference(m, p, hard, ns=5):
    sp = S.Space(S.Mesh(inputs.unit_sphere_patches(), m), p, continuous=hard)
    x = inputs.random_complex(sp.N, seed=5, cols=2)
    return x, A.cfie_matrix(sp, KAPPA, ETA, hard) @ x


def compare(m, p, hard, tol, **options):
    x, ref = reference(m, p, hard, options.get("gauss_singular", 5))
    prob, _ = G.problem(level_m=m, degree_p=p, kappa=KAPPA, eta_cfie=ETA, bc=int(hard), no_fmm=1, **options)
    assert G.rel(B.igabem_matvec(prob, x), ref) < tol
    B.igabem_problem_destroy(prob)


@pytest.mark.parametrize("hard", [False, True])
@pytest.mark.parametrize("m,p", [(0, 4), (1, 4), (0, 5)])
def test_degrees_above_three(m, p, hard):
    compare(m, p, hard, 1e-10)


@pytest.mark.parametrize("hard", [False, True])
@pytest.mark.parametrize("p", [1, 2])
@pytest.mark.parametrize("ns", [3, 4, 6])
def test_other_singular_rules(monkeypatch, ns, p, hard):
    monkeypatch.setattr(A, "singular_blocks", functools.partial(A.singular_blocks, n=ns))
    compare(1, p, hard, 1e-10, gauss_singular=ns)


@pytest.mark.parametrize("precision,tol", [(B.FP64, 1e-10), (B.MIXED_FP32, 2e-6)])
@pytest.mark.parametrize("m,p", [(0, 1), (1, 1), (2, 1), (0, 2), (1, 2), (2, 2)])
def test_sound_hard_regular_pairs(m, p, precision, tol):
    compare(m, p, True, tol, precision=precision)

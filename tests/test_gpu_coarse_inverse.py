"""The blocked Gauss-Jordan inverse of the coarsest system at its edges: one V-cycle against the
oracle with coarsest levels of 64 unknowns (two whole blocks), 169 (a remainder), 961 and 1089
(one and two rows per thread of the panel), 1681 (a narrower block), and the augmented system.

Bound: the dense inverse is good to about eps cond(A), cond(A) below 0.5 n_c^2 on n_c cells per
axis; with n_c <= 41 and a factor 100 for the elimination that is 1e-11 in FP64 and, with the
FP32 cycle's own rounding, 1e-4 in FP32."""
import numpy as np
import pytest

import workloads as W
from oracle.problem import OracleProblem
from tests.gpu_helpers import dev, gpu_problem, need_gpu, rel_err

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env():
    return need_gpu()


def interface(n):
    return W.ProblemSpec(n=n, geometry=W.Geometry(W.CIRCLE, (0.01, -0.02, 0.5), False), bc=W.INTERFACE, order=4,
                         box_bc=W.BOX_DIRICHLET, solution=W.two_phase_star_solution())


def pure_neumann(n):
    return W.ProblemSpec(n=n, geometry=W.Geometry(W.CIRCLE, (0.01, -0.02, 0.6), True), bc=W.NEUMANN, order=4,
                         solution=W.harmonic_exp_sin())


@pytest.mark.parametrize("case,n", [(interface, 64), (interface, 52), (interface, 62), (interface, 66), (interface, 82),
                                    (pure_neumann, 52), (pure_neumann, 48)])
def test_vcycle_with_the_coarse_inverse(env, case, n):
    torch, iim = env
    spec = case(n)
    O = OracleProblem(spec)
    v = np.random.default_rng(n).standard_normal(O.unk_flat.size) * O.unk_flat
    ref = O.precondition(v)
    for prec, tol in ((iim.MG_FP64, 1e-11), (iim.MG_FP32, 1e-4)):
        P = gpu_problem(iim, spec, mg_precision=prec)
        for _ in range(2):                     # a set-up re-run in place gives the same inverse
            assert rel_err(P.precondition(dev(v)).cpu().numpy(), ref) < tol
            P.setup()
        assert P.status() == 0

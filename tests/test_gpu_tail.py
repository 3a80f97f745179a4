"""The coarse tail, alone and as a cluster that shares the dense solve: one V- or W-cycle against the
oracle, for coarsest levels on both sides of the cluster's lines (100 nodes in FP64, 200 in FP32), one
level to three in the tail, in 2D and 3D and for every condition; the irregular rows of every level
come from the grouped set-up kernel.

Bounds: the oracle's own parity bounds, 1e-12 of the largest value in FP64, 1e-5 in FP32."""
import numpy as np
import pytest

import workloads as W
from oracle.problem import OracleProblem
from tests.gpu_helpers import dev, gpu_problem, need_gpu, rel_err

pytestmark = pytest.mark.gpu


def spec_of(dim, n, bc):
    body = W.CIRCLE if dim == 2 else W.SPHERE
    c = (0.013, -0.021, 0.017)[:dim]
    inside = bc == W.DIRICHLET
    sol = W.piecewise_polynomial(dim, 3, np.random.default_rng(n))
    return W.ProblemSpec(n=n, geometry=W.Geometry(body, (*c, 0.46), inside), bc=bc, order=4,
                         box_bc=W.BOX_NONE if inside else W.BOX_DIRICHLET, beta_plus=1.5,
                         beta_minus=0.5 if bc == W.INTERFACE else 1.0, solution=sol)


@pytest.fixture(scope="module")
def env():
    return need_gpu()


# coarsest level: 8^2 = 64 (alone), 11^2 = 121 (FP64 cluster), 15^2 = 225 (both); 5^3 = 125, 6^3 = 216, 9^3 = 729
@pytest.mark.parametrize("cycle", [1, 2])
@pytest.mark.parametrize("dim,n,bc", [(2, 64, W.NEUMANN), (2, 88, W.INTERFACE), (2, 60, W.NEUMANN),
                                      (2, 120, W.DIRICHLET), (3, 40, W.NEUMANN), (3, 48, W.DIRICHLET),
                                      (3, 36, W.INTERFACE)])
def test_cycle_matches_the_oracle(env, dim, n, bc, cycle):
    torch, iim = env
    spec = spec_of(dim, n, bc)
    O = OracleProblem(spec, cycle=cycle)
    v = np.random.default_rng(n).standard_normal(O.unk_flat.size) * O.unk_flat
    ref = O.precondition(v)
    for prec, tol in ((iim.MG_FP64, 1e-12), (iim.MG_FP32, 1e-5)):
        P = gpu_problem(iim, spec, mg_precision=prec, cycle=cycle)
        assert rel_err(P.precondition(dev(v)).cpu().numpy(), ref) < tol

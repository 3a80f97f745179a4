"""A cycle without pre-smoothing or without post-smoothing: the first visit of each level starts from u = 0
whether or not a sweep writes it.  V- and W-cycles with the finest level in the coarse tail, one level and
more above it, in 2D and 3D, against the oracle; the same bits from call to call.

Bounds: the oracle's own parity bounds, 1e-12 of the largest value in FP64, 1e-5 in FP32."""
import numpy as np
import pytest

import workloads as W
from oracle.problem import OracleProblem
from tests.gpu_helpers import dev, gpu_problem, need_gpu, rel_err

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env():
    return need_gpu()


@pytest.mark.parametrize("dim,n,bc", [(2, 32, W.DIRICHLET), (2, 64, W.NEUMANN), (2, 104, W.INTERFACE),
                                      (3, 20, W.DIRICHLET), (3, 40, W.NEUMANN)])
@pytest.mark.parametrize("nu1,nu2", [(0, 2), (0, 1), (2, 0)])
@pytest.mark.parametrize("cycle", [1, 2])
def test_cycle_matches_the_oracle(env, dim, n, bc, nu1, nu2, cycle):
    torch, iim = env
    inside = bc == W.DIRICHLET
    spec = W.ProblemSpec(n=n, geometry=W.Geometry(W.CIRCLE if dim == 2 else W.SPHERE,
                                                  ((0.013, -0.021, 0.017)[:dim] + (0.46,)), inside), bc=bc, order=4,
                         box_bc=W.BOX_NONE if inside else W.BOX_DIRICHLET, beta_plus=1.5,
                         beta_minus=0.5 if bc == W.INTERFACE else 1.0)
    O = OracleProblem(spec, nu1=nu1, nu2=nu2, cycle=cycle)
    v = np.random.default_rng(n).standard_normal(O.unk_flat.size) * O.unk_flat
    ref = O.precondition(v)
    for prec, tol in ((iim.MG_FP64, 1e-12), (iim.MG_FP32, 1e-5)):
        P = gpu_problem(iim, spec, mg_precision=prec, nu1=nu1, nu2=nu2, cycle=cycle)
        z = P.precondition(dev(v))
        assert rel_err(z.cpu().numpy(), ref) < tol
        # what another problem leaves in shared memory is not read
        gpu_problem(iim, spec, mg_precision=prec).precondition(dev(1e3 * v))
        assert torch.equal(P.precondition(dev(v)), z)


def test_nodes_between_walls_on_every_side(env):
    """A slender tilted body whose coarse levels hold nodes with no neighbour in phase (zero Neumann rows, no
    sweep moves them) under parents that have some: their right-hand side is a residual of either colour."""
    torch, iim = env
    spec = W.ProblemSpec(n=512, geometry=W.Geometry(W.ELLIPSE, (-0.1368, 0.0766, 0.3189, 0.0827, 0.297), True),
                         bc=W.NEUMANN, order=4, box_bc=W.BOX_NONE)
    O = OracleProblem(spec)
    zero = [(L.n, i % L.n + i // L.n) for L in O.mg.levels[:-1] if L.n <= 32
            for i in np.nonzero(L.unk_flat & (L.diag == 0))[0]]
    assert any(s % 2 for _, s in zero)                 # black, on a level of the tail
    v = np.random.default_rng(1).standard_normal(O.unk_flat.size) * O.unk_flat
    ref = O.precondition(v)
    for prec, tol in ((iim.MG_FP64, 1e-12), (iim.MG_FP32, 1e-5)):
        P = gpu_problem(iim, spec, mg_precision=prec)
        assert rel_err(P.precondition(dev(v)).cpu().numpy(), ref) < tol

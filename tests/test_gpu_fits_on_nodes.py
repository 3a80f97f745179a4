"""Bodies through grid nodes: a control point that sits exactly on a node has, for the side the node is not on,
several neighbours of that node as its nearest ones, and leaves out the one of the smallest index.  The
operator on random input against the oracle, whose rows tell which node was left out.  Circles have one such
neighbour; the dents of the star have three at the same distance, points of the sphere up to three.

Nodes lie exactly on the tangent at such a point, so a last bit of the point decides whether a set holds them:
the oracle's fits are built from the GPU's points and normals.

Bound: 3e-12 of the largest value, the parity bound of random input for such geometry."""
import numpy as np
import pytest

import workloads as W
from oracle.problem import OracleProblem
from tests.gpu_helpers import dev, gpu_problem, need_gpu, rel_err

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env():
    return need_gpu()


def dented(m):
    """r = 0.375 exactly, and least, at theta = 0."""
    return lambda n: W.Geometry(W.STAR, (1.0 / n, 1.0 / n, 0.4375, 0.0625, float(m), -np.pi / 2), False)


CASES = {
    "circle_4": (2, 4, 64, lambda n: W.Geometry(W.CIRCLE, (1.0 / n, 1.0 / n, 0.5), False)),
    "circle_6": (2, 6, 128, lambda n: W.Geometry(W.CIRCLE, (1.0 / n, 1.0 / n, 0.5), False)),
    "dents_4": (2, 4, 128, dented(4)),
    "dents_6": (2, 6, 256, dented(5)),
    "sphere_4": (3, 4, 32, lambda n: W.Geometry(W.SPHERE, (1.0 / n,) * 3 + (0.4375,), False)),
}


@pytest.mark.parametrize("case", sorted(CASES))
@pytest.mark.parametrize("bc", [W.INTERFACE, W.NEUMANN])
def test_operator_matches_the_oracle(env, case, bc):
    torch, iim = env
    dim, order, n, geometry = CASES[case]
    spec = W.ProblemSpec(n=n, geometry=geometry(n), bc=bc, order=order, box_bc=W.BOX_DIRICHLET, beta_plus=1.5,
                         beta_minus=0.5 if bc == W.INTERFACE else 1.0)
    O = OracleProblem(spec)
    P = gpu_problem(iim, spec)
    xc, nc = (a.cpu().numpy() for a in P.control_points())
    ax, lo, _ = (a.cpu().numpy() for a in P.control_point_edges())
    assert np.array_equal(ax, O.op.cross.axis) and np.array_equal(lo, O.op.cross.lo)
    pos = (xc + 1.0) * n / 2 - 0.5
    assert np.any(np.all(pos == np.round(pos), axis=1))
    O.op.cross.x[:], O.op.cross.normal[:] = xc, nc
    O.op._build_fits()
    u = np.random.default_rng(n).standard_normal(n ** dim) * O.unk_flat
    assert rel_err(P.apply(dev(u)).cpu().numpy(), O.op.apply(u)) < 3e-12

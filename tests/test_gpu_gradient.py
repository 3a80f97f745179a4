"""The gradient's node kernel against the oracle, with data, on random input: plain, box and affected nodes of
grids whose node count is and is not a multiple of a block's (256 nodes in 2D, 1024 in 3D), both orders, every
condition in 2D and 3D; zero at nodes that are no unknowns.

Bound: 1e-11 of the largest value, the gradient's parity bound."""
import numpy as np
import pytest

import workloads as W
from oracle.problem import OracleProblem
from tests.gpu_helpers import dev, gpu_problem, need_gpu, rel_err, set_gpu_data

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env():
    return need_gpu()


@pytest.mark.parametrize("dim,order,n,bc", [(2, 4, 40, W.DIRICHLET), (2, 4, 61, W.NEUMANN), (2, 4, 64, W.INTERFACE),
                                            (2, 6, 64, W.INTERFACE), (2, 6, 74, W.NEUMANN), (2, 6, 61, W.DIRICHLET),
                                            (3, 4, 32, W.DIRICHLET), (3, 4, 40, W.NEUMANN), (3, 4, 44, W.INTERFACE)])
def test_matches_the_oracle(env, dim, order, n, bc):
    torch, iim = env
    inside = bc == W.DIRICHLET
    spec = W.ProblemSpec(n=n, geometry=W.Geometry(W.CIRCLE if dim == 2 else W.SPHERE,
                                                  ((0.013, -0.021, 0.017)[:dim] + (0.46,)), inside), bc=bc, order=order,
                         box_bc=W.BOX_NONE if inside else W.BOX_DIRICHLET, beta_plus=1.5,
                         beta_minus=0.5 if bc == W.INTERFACE else 1.0,
                         solution=W.piecewise_polynomial(dim, 3, np.random.default_rng(n)))
    P = gpu_problem(iim, spec)
    set_gpu_data(P, spec)
    O = OracleProblem(spec)
    u = np.random.default_rng(1).standard_normal(n ** dim) * O.unk_flat
    g = P.gradient(dev(u)).cpu().numpy()
    assert rel_err(g, O.op.gradient(u, O.data()[1])) < 1e-11
    assert np.all(g[:, ~O.unk_flat.astype(bool)] == 0)

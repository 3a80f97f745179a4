"""The operator's two launches against the batched engine's three kernels and the oracle: plain and
affected nodes at the grid's edges, for grids whose node count is and is not a multiple of a block,
in 2D and 3D; the right-hand side and the gradient, which share the node classes.

Bound: 1e-12 of the largest value (the operator's parity bound), 1e-11 for the gradient."""
import numpy as np
import pytest

import workloads as W
from oracle.problem import OracleProblem
from tests.gpu_helpers import dev, gpu_problem, need_gpu, rel_err, set_gpu_data

pytestmark = pytest.mark.gpu


def spec_of(dim, order, n, bc):
    body = W.CIRCLE if dim == 2 else W.SPHERE
    c = (0.013, -0.021, 0.017)[:dim]
    inside = bc == W.DIRICHLET
    sol = W.piecewise_polynomial(dim, 3, np.random.default_rng(n))
    return W.ProblemSpec(n=n, geometry=W.Geometry(body, (*c, 0.46), inside), bc=bc, order=order,
                         box_bc=W.BOX_NONE if inside else W.BOX_DIRICHLET, beta_plus=1.5,
                         beta_minus=0.5 if bc == W.INTERFACE else 1.0, solution=sol)


@pytest.fixture(scope="module")
def env():
    return need_gpu()


@pytest.mark.parametrize("dim,order,n,bc", [(2, 4, 40, W.DIRICHLET), (2, 4, 61, W.NEUMANN), (2, 6, 64, W.INTERFACE),
                                            (2, 6, 74, W.NEUMANN), (3, 4, 40, W.NEUMANN), (3, 4, 44, W.INTERFACE)])
def test_apply_rhs_and_gradient(env, dim, order, n, bc):
    torch, iim = env
    spec = spec_of(dim, order, n, bc)
    P = gpu_problem(iim, spec)
    f = set_gpu_data(P, spec)
    O = OracleProblem(spec)
    u = np.random.default_rng(1).standard_normal(n ** dim) * O.unk_flat
    w = P.apply(dev(u)).cpu().numpy()
    assert rel_err(w, O.op.apply(u)) < 3e-12
    assert np.all(w[~O.unk_flat.astype(bool)] == 0)
    assert np.array_equal(P.apply_noalloc(dev(u)).cpu().numpy(), w)
    # b = f - (operator of 0 with the data)
    lg = P.apply(dev(np.zeros_like(u)), include_data=True).cpu().numpy()
    assert rel_err(P.rhs().cpu().numpy(), (f - lg) * O.unk_flat) < 1e-14

"""The least-squares fits on both of their kernels: piecewise polynomials of the scheme's
degree are reproduced by the operator with data, for bodies whose control points are all
ordinary and for bodies through grid nodes, whose control points sit exactly on the far node
of one side (the fits that the common-case kernel leaves to the CTA kernel).

Bound: the operator's own rounding.  A row sums the stencil (coefficients of size n^2 / 4 per
axis, sum of magnitudes below 11) over u and over ghosts whose least-squares rows have sums of
magnitudes below 45, so 500 eps d (n/2)^2 max|u| covers it."""
import numpy as np
import pytest

import workloads as W
from tests.gpu_helpers import dev, gpu_problem, need_gpu, set_gpu_data

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env():
    return need_gpu()


def spec_of(dim, order, n, bc, on_node, seed):
    h = 2.0 / n
    c = [h / 2] * dim if on_node else [0.013, -0.021, 0.017][:dim]
    r = (n // 4) * h if on_node else 0.47
    rng = np.random.default_rng(seed)
    g = W.Geometry(W.CIRCLE if dim == 2 else W.SPHERE, (*c, r), bc == W.DIRICHLET)
    return W.ProblemSpec(n=n, geometry=g, bc=bc, order=order, box_bc=W.BOX_NONE if bc == W.DIRICHLET else W.BOX_DIRICHLET,
                         beta_plus=1.5, beta_minus=1.0 if bc != W.INTERFACE else 0.5,
                         solution=W.piecewise_polynomial(dim, order, rng))


@pytest.mark.parametrize("on_node", [False, True])
@pytest.mark.parametrize("bc", [W.DIRICHLET, W.NEUMANN, W.INTERFACE])
@pytest.mark.parametrize("dim,order,n", [(2, 4, 48), (2, 6, 64), (2, 6, 100), (3, 4, 48)])
def test_polynomials_reproduced(env, dim, order, n, bc, on_node):
    spec = spec_of(dim, order, n, bc, on_node, 10 * n + bc)
    P = gpu_problem(env[1], spec)
    f = set_gpu_data(P, spec)
    X = W.node_coords(n, dim)
    phase = W.from_flat(P.phase().cpu().numpy().astype(bool), n, dim)
    s = spec.solution
    u = np.where(phase, s.u_plus(X), s.u_minus(X) if bc == W.INTERFACE else 0.0)
    w = P.apply(dev(W.to_flat(u)), include_data=True).cpu().numpy()
    assert np.max(np.abs(w - f)) <= 500 * 2.0 ** -53 * dim * (n / 2) ** 2 * 1.5 * np.max(np.abs(u))

"""The 3D half sweeps that take two pairs through several planes (levels that exceed L2, from 204^3 on):
bit for bit the separate kernels of the batched engine, in runs that end inside and at the grid's edge,
with box faces, irregular rows and cells that are no unknowns in one pair."""
import numpy as np
import pytest

import workloads as W
from tests.gpu_helpers import gpu_problem, need_gpu, set_gpu_data

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env():
    return need_gpu()


@pytest.mark.parametrize("n,bc", [(208, W.NEUMANN), (224, W.DIRICHLET), (208, W.INTERFACE)])
def test_same_bits_as_the_separate_kernels(env, n, bc):
    torch, iim = env
    inside = bc == W.DIRICHLET
    spec = W.ProblemSpec(n=n, geometry=W.Geometry(W.SPHERE, (0.013, -0.021, 0.017, 0.46), inside), bc=bc, order=4,
                         box_bc=W.BOX_NONE if inside else W.BOX_DIRICHLET, beta_plus=1.5,
                         beta_minus=0.5 if bc == W.INTERFACE else 1.0,
                         solution=W.piecewise_polynomial(3, 3, np.random.default_rng(n)))
    P = gpu_problem(iim, spec)
    set_gpu_data(P, spec)
    x, info = P.solve()
    E = iim.Engine(iim.default_options(), 2)
    slot = E.admit(P)
    E.solve_all()
    y = torch.empty_like(x)
    got = E.release(slot, y)
    assert info.converged and got.iters == info.iters
    assert torch.equal(x, y)

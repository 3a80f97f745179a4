"""The 3D multigrid kernels (a launch per half sweep and transfer, u and f stored by colour): one V-cycle
against the oracle, and bit for bit the separate kernels of the batched engine, for sizes with one to
four levels above the tail, rows that are and are not whole warps, and every condition.

Bound for FP64: the oracle's own parity bound, 1e-12 of the largest value."""
import numpy as np
import pytest

import workloads as W
from oracle.problem import OracleProblem
from tests.gpu_helpers import dev, gpu_problem, need_gpu, rel_err, set_gpu_data

pytestmark = pytest.mark.gpu

BODIES = {
    "dirichlet": lambda n: W.ProblemSpec(
        n=n, geometry=W.Geometry(W.SPHERE, (0.02, -0.01, 0.03, 0.6), True), bc=W.DIRICHLET, order=4,
        solution=W.sin_sin_cos_3d((1.0, 2.0, 1.5), (0.1, 0.2, 0.3))),
    "neumann": lambda n: W.ProblemSpec(
        n=n, geometry=W.Geometry(W.SPHERE, (0.02, -0.01, 0.03, 0.45), False), bc=W.NEUMANN, order=4,
        box_bc=W.BOX_DIRICHLET, beta_plus=2.0, solution=W.sin_sin_cos_3d((1.0, 2.0, 1.5), (0.1, 0.2, 0.3))),
    "interface": lambda n: W.ProblemSpec(
        n=n, geometry=W.Geometry(W.SPHERE, (0.02, -0.01, 0.03, 0.45), False), bc=W.INTERFACE, order=4,
        box_bc=W.BOX_DIRICHLET, beta_plus=1.0, beta_minus=2.0,
        solution=W.piecewise_polynomial(3, 4, np.random.default_rng(5))),
}


@pytest.fixture(scope="module")
def env():
    return need_gpu()


@pytest.mark.parametrize("body,n", [("dirichlet", 32), ("neumann", 40), ("interface", 40)])
def test_vcycle_matches_the_oracle(env, body, n):
    torch, iim = env
    spec = BODIES[body](n)
    O = OracleProblem(spec)
    v = np.random.default_rng(n).standard_normal(O.unk_flat.size) * O.unk_flat
    ref = O.precondition(v)
    for prec, tol in ((iim.MG_FP64, 1e-12), (iim.MG_FP32, 1e-5)):
        P = gpu_problem(iim, spec, mg_precision=prec)
        assert rel_err(P.precondition(dev(v)).cpu().numpy(), ref) < tol


@pytest.mark.parametrize("body,n,prec", [("dirichlet", 24, 0), ("dirichlet", 56, 0), ("neumann", 64, 0),
                                         ("interface", 96, 0), ("neumann", 48, 2), ("dirichlet", 112, 0),
                                         ("neumann", 160, 0)])
def test_same_bits_as_the_separate_kernels(env, body, n, prec):
    torch, iim = env
    spec = BODIES[body](n)
    P = gpu_problem(iim, spec, mg_precision=prec)
    set_gpu_data(P, spec)
    x, info = P.solve()
    E = iim.Engine(iim.default_options(mg_precision=prec), 2)
    slot = E.admit(P)
    E.solve_all()
    y = torch.empty_like(x)
    einfo = E.release(slot, y)
    assert einfo.iters == info.iters
    assert torch.equal(x, y)

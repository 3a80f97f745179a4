"""3D levels that exceed L2, in the forms of the multigrid precision: FP64 (a plane per thread) against FP32
(runs of planes), and BF16 right-hand sides below the finest level, where a run reads them in pairs, bit for
bit the separate kernels of the batched engine after three iterations.

Bound FP32 / FP64: the sum of both forms' parity bounds against the oracle, 1e-5 and 1e-12 of the largest value."""
import numpy as np
import pytest

import workloads as W
from tests.gpu_helpers import gpu_problem, need_gpu

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env():
    return need_gpu()


def spec_of(n, bc):
    inside = bc == W.DIRICHLET
    return W.ProblemSpec(n=n, geometry=W.Geometry(W.SPHERE, (0.013, -0.021, 0.017, 0.46), inside), bc=bc, order=4,
                         box_bc=W.BOX_NONE if inside else W.BOX_DIRICHLET, beta_plus=1.5,
                         beta_minus=0.5 if bc == W.INTERFACE else 1.0)


@pytest.mark.parametrize("n,bc", [(208, W.NEUMANN), (224, W.DIRICHLET)])
def test_fp64_and_fp32_agree(env, n, bc):
    torch, iim = env
    spec, z = spec_of(n, bc), []
    v = torch.randn(n ** 3, dtype=torch.float64, device="cuda", generator=torch.Generator("cuda").manual_seed(n))
    for prec in (iim.MG_FP64, iim.MG_FP32):
        P = gpu_problem(iim, spec, mg_precision=prec)
        z.append(P.precondition(v * P.phase()))
        del P
    assert float((z[0] - z[1]).abs().max() / z[0].abs().max()) < 1e-5 + 1e-12


def test_bf16_right_hand_sides(env):
    torch, iim = env
    n = 416                                            # the level below has 208^3 cells
    opts = dict(mg_precision=iim.MG_FP32_BF16R, max_iter=3)
    P = gpu_problem(iim, spec_of(n, W.NEUMANN), **opts)
    f = torch.randn(n ** 3, dtype=torch.float64, device="cuda", generator=torch.Generator("cuda").manual_seed(n))
    zero = torch.zeros
    P.set_data(f, zero(P.K, dtype=torch.float64, device="cuda"), None, None,
               zero(P.B, dtype=torch.float64, device="cuda"))
    x, info = P.solve(check=False)
    assert info.iters == 3 and x.abs().max() > 0
    E = iim.Engine(iim.default_options(**opts), 1)
    slot = E.admit(P)
    E.solve_all()
    y = torch.empty_like(x)
    got = E.release(slot, y, check=False)
    assert got.iters == 3
    assert torch.equal(x, y)

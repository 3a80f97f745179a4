"""Vectors that start between two pairs of doubles (a contiguous slice t[1:]): each call that takes device
vectors gives the bits it gives for aligned ones."""
import ctypes

import numpy as np
import pytest

import workloads as W
from tests.gpu_helpers import dev, gpu_data, gpu_problem, need_gpu

pytestmark = pytest.mark.gpu


def spec_of(dim, n):
    return W.ProblemSpec(n=n, geometry=W.Geometry(W.CIRCLE if dim == 2 else W.SPHERE,
                                                  ((0.013, -0.021, 0.017)[:dim] + (0.46,)), False), bc=W.NEUMANN,
                         order=4, box_bc=W.BOX_DIRICHLET, solution=W.piecewise_polynomial(dim, 3, np.random.default_rng(n)))


@pytest.fixture(scope="module")
def env():
    return need_gpu()


# the coarse tail alone, one kernel per step, two, the 3D kernels, those of levels that exceed L2; sweeps (1, 1)
# take the generic 2D kernels
@pytest.mark.parametrize("dim,n,nu", [(2, 32, 2), (2, 64, 2), (2, 128, 2), (2, 128, 1), (3, 40, 2), (3, 208, 2)])
@pytest.mark.parametrize("prec", [0, 1])
def test_precondition(env, dim, n, nu, prec):
    torch, iim = env
    P = gpu_problem(iim, spec_of(dim, n), mg_precision=prec, nu1=nu, nu2=nu)
    lib, N = iim.load(), P.N
    v = dev(np.random.default_rng(n).standard_normal(N))
    ref = P.precondition(v)
    big = torch.full((N + 2,), -7.0, dtype=torch.float64, device="cuda")
    vin = torch.empty(N + 1, dtype=torch.float64, device="cuda")
    vin[1:] = v
    odd_v, odd_z = vin[1:], big[1:N + 1]
    assert odd_v.data_ptr() % 16 == 8 and odd_z.data_ptr() % 16 == 8 and v.data_ptr() % 16 == 0
    assert torch.equal(P.precondition(odd_v), ref)
    for a in (v, odd_v):
        odd_z.zero_()
        assert lib.iim_precondition(P.h, ctypes.c_void_p(a.data_ptr()), ctypes.c_void_p(odd_z.data_ptr())) == 0
        assert torch.equal(odd_z, ref) and big[0] == -7.0 and big[-1] == -7.0
        assert torch.equal(a, v)


@pytest.mark.parametrize("dim,n", [(2, 64), (3, 40), (3, 96)])
def test_operator_and_solve(env, dim, n):
    torch, iim = env
    spec = spec_of(dim, n)
    P = gpu_problem(iim, spec)
    odd = lambda a: torch.cat([torch.zeros(1, dtype=torch.float64, device="cuda"), dev(a)])[1:]
    data = [x for x in gpu_data(P, spec)]
    out = []
    for put in (dev, odd):
        P.set_data(*[None if x is None else put(x) for x in data])
        u = put(np.random.default_rng(n).standard_normal(P.N))
        out.append([P.rhs(), P.apply(u), P.apply(u, include_data=True), P.gradient(u), P.boundary_values(u), P.solve()[0]])
    for a, b in zip(*out):
        assert torch.equal(a, b)

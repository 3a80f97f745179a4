"""The operator's fixed-point tiles (3D grids of 2^19 nodes and more) against the exact sum at plain
nodes, for tiles cut by the grid's edge (and one 2D grid, which has none): smooth u, random u, u over
100 binades (where nodes and tiles are left to the FP64 sum), zeros, and a NaN or an infinity, which
may reach only the nodes whose stencil holds it.  The batched engine's tiles give the same bits.

Bound on the error: 16 rounding errors of the stencil's absolute coefficients times its largest value,
13 terms summed in FP64; the tiles' cut is below 1.5 2^-54 of the same product."""
import numpy as np
import pytest

import workloads as W
from tests.gpu_helpers import dev, gpu_problem, need_gpu, set_gpu_data

pytestmark = pytest.mark.gpu
COEF = {4: (np.longdouble(16) / 12, np.longdouble(-1) / 12),
        6: (np.longdouble(270) / 180, np.longdouble(-27) / 180, np.longdouble(2) / 180)}
GRIDS = [(2, 6, 736, W.INTERFACE), (3, 4, 88, W.DIRICHLET), (3, 4, 88, W.INTERFACE), (3, 4, 104, W.NEUMANN)]


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


def shifted(a, ax, j, fill):
    out = np.full_like(a, fill)
    src, dst = [slice(None)] * a.ndim, [slice(None)] * a.ndim
    src[ax], dst[ax] = (slice(j, None), slice(None, -j)) if j > 0 else (slice(None, j), slice(-j, None))
    out[tuple(dst)] = a[tuple(src)]
    return out


def reference(u, phase, coef, unknown):
    """exact sum, largest |u| in the stencil, plain nodes; arrays [z, y, x]"""
    d = u.ndim
    U = u.astype(np.longdouble)
    s, big, plain = -2 * d * sum(coef) * U, np.abs(u), unknown.copy()
    for ax in range(d):
        for j, a in enumerate(coef, 1):
            for sj in (-j, j):
                s = s + a * shifted(U, ax, sj, 0)
                big = np.maximum(big, shifted(np.abs(u), ax, sj, 0))
                plain &= shifted(phase.astype(int), ax, sj, -1) == phase
    return s, big, plain


@pytest.mark.parametrize("dim,order,n,bc", GRIDS)
def test_plain_nodes(env, dim, order, n, bc):
    torch, iim = env
    spec = spec_of(dim, order, n, bc)
    P = gpu_problem(iim, spec)
    shape = (n,) * dim
    phase = P.phase().cpu().numpy().reshape(shape).astype(bool)
    unknown = np.ones(shape, bool) if bc == W.INTERFACE else phase
    beta = np.where(phase, spec.beta_plus, spec.beta_minus if bc == W.INTERFACE else 1.0)
    coef = COEF[order]
    rng = np.random.default_rng(2)
    x = np.meshgrid(*[np.arange(n) / n] * dim, indexing="ij")
    smooth = sum(np.sin(5 * a + k) for k, a in enumerate(x))
    wide = rng.standard_normal(shape) * 2.0 ** rng.integers(-50, 50, shape)
    amp = sum(abs(2 * a) for a in coef) * 2 * dim
    factor = None
    for u in (smooth, rng.standard_normal(shape), wide):
        w = P.apply(dev((u * unknown).reshape(-1))).cpu().numpy().reshape(shape)
        s, big, plain = reference(u * unknown, phase, coef, unknown)
        if factor is None:                        # 1 / h^2 from the smooth field
            factor = np.float64((w[plain] * s[plain]).sum() / (beta[plain] * s[plain] ** 2).sum())
            factor = round(factor * 64) / 64
        err = np.abs(w[plain] - factor * beta[plain] * s[plain])
        assert np.all(err <= 16 * 2.0 ** -53 * amp * factor * beta[plain] * big[plain])
    # values at nodes that are no unknowns take no part
    junk = np.where(unknown, smooth, np.nan)
    a = P.apply(dev(junk.reshape(-1))).cpu().numpy().reshape(shape)
    b = P.apply(dev((smooth * unknown).reshape(-1))).cpu().numpy().reshape(shape)
    assert np.array_equal(a[plain], b[plain])
    # zeros, and one value that is no number: only the nodes that read it change
    assert np.all(P.apply(dev(np.zeros(n ** dim))).cpu().numpy() == 0)
    at = tuple(v[len(v) // 2] for v in np.nonzero(plain))
    for bad in (np.nan, np.inf, 1e300):
        u = smooth * unknown
        u[at] = bad
        w = P.apply(dev(u.reshape(-1))).cpu().numpy().reshape(shape)
        near = np.zeros(shape, bool)
        near[at] = True
        reads = near.copy()
        for ax in range(dim):
            for j in range(1, len(coef) + 1):
                reads |= shifted(near, ax, j, False) | shifted(near, ax, -j, False)
        assert not np.any(np.isfinite(w[reads & plain])) or bad == 1e300
        s, big, _ = reference(smooth * unknown, phase, coef, unknown)
        keep = plain & ~reads
        err = np.abs(w[keep] - factor * beta[keep] * s[keep])
        assert np.all(err <= 16 * 2.0 ** -53 * amp * factor * beta[keep] * big[keep])


def test_engine_tiles_have_the_same_bits(env):
    torch, iim = env
    for dim, order, n, bc in (GRIDS[1], GRIDS[3]):
        spec = spec_of(dim, order, n, bc)
        P = gpu_problem(iim, spec)
        set_gpu_data(P, spec)
        x, info = P.solve()
        E = iim.Engine(iim.default_options(), max_slots=4)
        Q = gpu_problem(iim, spec)
        set_gpu_data(Q, spec)
        slot = E.admit(Q)
        E.solve_all()
        y = torch.zeros(Q.N, dtype=torch.float64, device="cuda")
        got = E.release(slot, y)
        assert got.iters == info.iters and torch.equal(x, y)
        E.close()

"""The node count behind the benchmark's stencil roofline: the unknowns that the oracle's operator records touch
nowhere."""
import pytest

import bench
import workloads as W

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("dim,order,n,bc", [(2, 6, 64, W.INTERFACE), (2, 4, 48, W.DIRICHLET), (3, 4, 32, W.NEUMANN)])
def test_plain_nodes_match_the_oracle(dim, order, n, bc):
    from oracle.operator import IIMOperator
    inside = bc == W.DIRICHLET
    c = (0.01, -0.02, 0.03)[:dim] + (0.5 if dim == 2 else 0.4,)
    spec = W.ProblemSpec(n=n, geometry=W.Geometry(W.CIRCLE if dim == 2 else W.SPHERE, c, inside), bc=bc, order=order,
                         box_bc=W.BOX_NONE if inside else W.BOX_DIRICHLET)
    op = IIMOperator(spec)
    affected = {r[0] for r in op.iim_rec} | {r[0] for r in op.box_rec}
    phase = torch.from_numpy(op.plus.ravel(order="F").copy())
    assert bench.plain_nodes(phase, n, dim, order // 2, bc == W.INTERFACE) == int(op.unknown.sum()) - len(affected)

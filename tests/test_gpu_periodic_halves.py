"""Periodic levels that run by halves of the cycle, and first sweeps from a zero
iterate, against the same cycle launched step by step, bit for bit: each set of
periodic axes, sizes of one tile and of several, both stencil kinds, every sweep
count the tiles allow, as a stationary cycle and inside flexible CG."""
import numpy as np
import pytest
import torch

from test_gpu_periodic import hierarchy, problem

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("axes", ["x", "y", "xy"])
@pytest.mark.parametrize("n,kind,nu", [(15, 9, (2, 1)), (31, 9, (1, 1)), (63, 5, (2, 1)), (127, 9, (2, 2)),
                                       (255, 9, (1, 2)), (511, 9, (2, 1)), (511, 5, (2, 1)), (1023, 9, (2, 1))])
@pytest.mark.parametrize("krylov", ["none", "fcg"])
def test_periodic_halves_are_the_stepwise_cycle(bmg, axes, n, kind, nu, krylov):
    kind, planes, f, px, py = problem(n, axes, seed=80 + n, kind=kind)
    out = []
    for graph in (True, False):
        h = hierarchy(bmg, kind, planes, axes, use_graph=graph, nu1=nu[0], nu2=nu[1], krylov=krylov, arith="fused")
        x, it, rr, ok = h.solve(torch.from_numpy(f).cuda(), tol=0.0, maxit=3)
        out.append((x.cpu().numpy()[1:-1, 1:-1], h.history()))
        h.close()
    assert np.array_equal(out[0][0], out[1][0]) and out[0][1] == out[1][1]

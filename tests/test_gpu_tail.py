"""The level-fused tail against the same cycle launched step by step: every size
it can start at, coarsest levels it solves one lane per unknown and by the
general warp solve, sweep counts down to none, and a top level that starts from
a non-zero iterate.  Every value is one expression of the same operands, so the
two agree bit for bit."""
import numpy as np
import pytest
import torch

import workloads as w

pytestmark = pytest.mark.gpu


def solve_pair(bmg, kind, planes, f, cycles, **kw):
    coef = torch.from_numpy(planes[:3] if kind == 5 else planes).cuda()
    out = []
    for graph in (True, False):
        h = bmg.Hierarchy(kind, coef, use_graph=graph, **kw)
        x, it, rr, ok = h.solve(torch.from_numpy(f).cuda(), tol=0.0, maxit=cycles)
        out.append((x.cpu().numpy(), h.history(), h))
    return out


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("kind,n,coarsest,nu", [(9, 7, 3, (2, 1)), (9, 15, 3, (1, 2)), (9, 31, 7, (2, 1)),
                                                (9, 63, 15, (2, 1)), (5, 63, 3, (3, 0)), (5, 31, 3, (2, 1)),
                                                (9, 127, 3, (0, 3)), (9, 63, 3, (1, 1))])
@pytest.mark.parametrize("arith", ["rounded", "fused"])
def test_tail_is_the_stepwise_cycle(bmg, precision, kind, n, coarsest, nu, arith):
    planes = w.poisson5(n) if kind == 5 else w.fe9_from_cells(w.lognormal_cells(n, 2.0, 6.0, 60 + n))
    f = w.rhs_uniform(n, 61 + n)
    a, b = solve_pair(bmg, kind, planes, f, 3, precision=precision, coarsest=coarsest, nu1=nu[0], nu2=nu[1],
                      arith=arith, inner_cycles=2 if precision == "fp32" else 1)
    assert np.array_equal(a[0], b[0]) and a[1] == b[1]

"""Cycles whose level 0 is where the level-fused tail starts, with a sweep kernel
forced on it that would not read a zero iterate: the tail reads one, so it has to
be there.  Against the same cycle launched step by step, bit for bit, over more
steps than one (the first starts from zeros in any case)."""
import numpy as np
import pytest
import torch

import workloads as w

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("smoother", ["rows", "tile0", "tile3", "tile5", "pair0", "pair3"])
@pytest.mark.parametrize("n,krylov,inner,nu", [(63, "none", 1, (2, 1)), (31, "none", 2, (2, 2)), (15, "none", 1, (1, 1)),
                                               (63, "fcg", 1, (2, 1)), (31, "fcg", 2, (3, 1))])
@pytest.mark.parametrize("precision", ["fp32", "bf16"])
def test_forced_sweeps_above_the_tail(bmg, smoother, n, krylov, inner, nu, precision):
    planes = w.fe9_from_cells(w.lognormal_cells(n, 1.5, 6.0, 90 + n))
    coef, f = torch.from_numpy(planes).cuda(), torch.from_numpy(w.rhs_uniform(n, 91 + n)).cuda()
    out = []
    for graph in (True, False):
        h = bmg.Hierarchy(9, coef, precision=precision, smoother=smoother, krylov=krylov, inner_cycles=inner,
                          nu1=nu[0], nu2=nu[1], use_graph=graph, arith="fused")
        x, it, rr, ok = h.solve(f, tol=0.0, maxit=4)
        out.append((x.cpu().numpy(), h.history()))
        h.close()
    assert np.array_equal(out[0][0], out[1][0]) and out[0][1] == out[1][1]
    assert out[0][1][-1] < 0.05 * out[0][1][0]

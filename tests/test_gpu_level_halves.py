"""Levels that run by halves (one launch down, one up) against the same cycle
launched step by step, bit for bit: grids of one tile and of several with ragged
last tiles, both stencil kinds and arithmetic modes, every sweep count the
tiles allow, and an embedded grid with identity rows."""
import numpy as np
import pytest
import torch

import workloads as w

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["fp64", "fp32", "bf16"])
@pytest.mark.parametrize("kind,nx,ny,nu", [(9, 31, 31, (2, 1)), (9, 127, 127, (1, 1)), (5, 127, 127, (2, 1)),
                                           (9, 255, 255, (2, 2)), (9, 511, 511, (2, 1)), (5, 255, 255, (1, 2)),
                                           (9, 300, 200, (2, 1)), (9, 1023, 1023, (2, 1))])
@pytest.mark.parametrize("arith", ["rounded", "fused"])
def test_halves_are_the_stepwise_cycle(bmg, precision, kind, nx, ny, nu, arith):
    _, planes, f = w.general_size_problem(nx, ny, kind)
    coef = torch.from_numpy(planes[:3] if kind == 5 else planes).cuda()
    rhs = torch.from_numpy(f).cuda()
    out = []
    for graph in (True, False):
        h = bmg.Hierarchy(kind, coef, precision=precision, nu1=nu[0], nu2=nu[1], arith=arith, use_graph=graph)
        before = h.launch_count
        x, it, rr, ok = h.solve(rhs, tol=0.0, maxit=3)
        out.append((x.cpu().numpy(), h.history(), h.launch_count - before))
        h.close()
    assert np.array_equal(out[0][0], out[1][0]) and out[0][1] == out[1][1]
    assert out[0][2] < out[1][2]        # fewer launches: the halves ran

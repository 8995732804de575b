"""Device memory of many small hierarchies.  A problem's arrays come to about 24
FP64 planes of its finest level (stencil 6, weights 2, FP32 copies, packed
stencils and iterates 10, a third more for the coarser levels) and some 50 KB
that do not depend on the size, a member of a batch of right-hand sides' to 3
planes; twice that is the bound, over a batch whose own tables are small."""
import pytest
import torch

import workloads as w

pytestmark = pytest.mark.gpu


def taken(make, count):
    make().close()                       # modules loaded, tuners warm
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    obj = make()
    torch.cuda.synchronize()
    got = before - torch.cuda.mem_get_info()[0]
    obj.close()
    return got / count


@pytest.mark.parametrize("precision", ["fp64", "fp32", "bf16"])
@pytest.mark.parametrize("n,count", [(7, 400), (15, 400), (31, 300), (63, 200)])
def test_small_problems_take_what_their_arrays_need(bmg, precision, n, count):
    coef = torch.from_numpy(w.fe9_from_cells(w.lognormal_cells(n, 1.0, 4.0, 40 + n))).cuda()
    plane = 8 * (n + 2) ** 2
    assert taken(lambda: bmg.Batch(9, [coef] * count, precision=precision), count) <= 2 * (24 * plane + 50 * 1024)
    h = bmg.Hierarchy(9, coef, precision=precision)
    assert taken(lambda: bmg.Batch.from_hierarchy(h, count), count) <= 2 * (3 * plane + 50 * 1024)
    h.close()


def test_a_periodic_hierarchy_takes_what_its_arrays_need(bmg):
    kind, planes, f, px, py = w.periodic_problem(1023, "x", std=1.0, corr_len=8.0)
    coef = torch.from_numpy(planes).cuda()
    # stencil 6, weights 2, residual, second iterate and, below the top, iterate and right-hand side
    arrays = (6 + 2 + 2 + 2) * 4 / 3 * 8 * 1026 * 1025
    assert taken(lambda: bmg.Hierarchy(kind, coef, periodic="x"), 1) <= arrays + (8 << 20)

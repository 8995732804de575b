"""Batched stages that run by halves, and batched pre-smoothing with the
restriction in the same pass, against the same cycles launched step by step, bit
for bit: uneven batches whose stages hold level-0 and coarse levels side by side,
grids narrower than one strip, both stencil kinds and arithmetic modes, one and
two inner cycles, and several right-hand sides of one operator."""
import pytest
import torch

import workloads as w

pytestmark = pytest.mark.gpu


def problems(sizes, kind):
    out = []
    for k, n in enumerate(sizes):
        _, planes, f = w.general_size_problem(n, n, kind)
        out.append((torch.from_numpy(planes[:3] if kind == 5 else planes).cuda().contiguous(),
                    torch.from_numpy(f).cuda() * (1.0 + 0.25 * k)))
    return out


def run(bmg, probs, kind, monkeypatch=None, fuse=0, **kw):
    if monkeypatch is not None:
        opts = bmg._lib.Opts

        def make(*a):
            o = opts(*a)
            o.fuse_restrict = fuse
            return o
        monkeypatch.setattr(bmg._lib, "Opts", make)
    B = bmg.Batch(kind, [p[0] for p in probs], **kw)
    if monkeypatch is not None:
        monkeypatch.undo()
    xs, its, rrs, ok = B.solve([p[1] for p in probs], tol=0.0, maxit=3)
    out = ([x.clone() for x in xs], [B.history(k) for k in range(len(probs))])
    B.close()
    return out


def same(a, b):
    return all(torch.equal(p, q) for p, q in zip(a[0], b[0])) and a[1] == b[1]


@pytest.mark.parametrize("precision", ["fp64", "fp32", "bf16"])
@pytest.mark.parametrize("kind,nu,inner", [(9, (2, 1), 1), (5, (2, 1), 2), (9, (1, 2), 2), (9, (2, 2), 1)])
@pytest.mark.parametrize("arith", ["rounded", "fused"])
def test_batched_halves_are_the_stepwise_cycle(bmg, precision, kind, nu, inner, arith):
    probs = problems([63, 255, 127, 31, 255, 63, 511], kind)
    kw = dict(precision=precision, nu1=nu[0], nu2=nu[1], inner_cycles=inner, arith=arith)
    assert same(run(bmg, probs, kind, use_graph=True, **kw), run(bmg, probs, kind, use_graph=False, **kw))


@pytest.mark.parametrize("precision", ["fp32", "bf16"])
@pytest.mark.parametrize("smoother", ["pair0", "pair3"])
@pytest.mark.parametrize("inner", [1, 2])
@pytest.mark.parametrize("arith", ["rounded", "fused"])
def test_batched_restriction_in_the_two_sweep_pass(bmg, monkeypatch, precision, smoother, inner, arith):
    probs = problems([63, 255, 7, 127, 15, 255, 31], 9)
    kw = dict(precision=precision, inner_cycles=inner, arith=arith, use_graph=False)
    one = run(bmg, probs, 9, monkeypatch, fuse=2, smoother=smoother, **kw)
    assert same(one, run(bmg, probs, 9, monkeypatch, fuse=1, smoother=smoother, **kw))
    assert same(one, run(bmg, probs, 9, **kw))


@pytest.mark.parametrize("precision", ["fp32", "bf16"])
@pytest.mark.parametrize("count", [1, 5])
def test_right_hand_sides_choose_either_pass(bmg, precision, count):
    coef, f = problems([1023], 9)[0]
    h = bmg.Hierarchy(9, coef, precision=precision, arith="fused")
    rhs = [f * (1.0 + k) for k in range(count)]
    out = []
    for graph in (True, False):
        B = bmg.Batch.from_hierarchy(h, count, use_graph=graph)
        xs, its, rrs, ok = B.solve(rhs, tol=0.0, maxit=3)
        out.append(([x.clone() for x in xs], [B.history(k) for k in range(count)]))
        B.close()
    h.close()
    assert same(out[0], out[1])

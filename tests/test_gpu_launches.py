"""Which launches an iteration is made of, counted on the library's own counter:
levels by halves are two launches each, the level-fused tail one, so that a rule
of choice that no longer picks them shows here (their results are the same bits
as the step-by-step cycle's either way)."""
import pytest
import torch

import workloads as w
from test_gpu_periodic import problem as periodic_problem

pytestmark = pytest.mark.gpu


def problem(n, kind=9):
    _, planes, f = w.general_size_problem(n, n, kind)
    return torch.from_numpy(planes[:3] if kind == 5 else planes).cuda().contiguous(), torch.from_numpy(f).cuda()


def batch_iteration(bmg, monkeypatch, probs, fuse=0, **kw):
    """Launches of one iteration, and the iterates and histories of four."""
    opts = bmg._lib.Opts

    def make(*a):
        o = opts(*a)
        o.fuse_restrict = fuse
        return o
    monkeypatch.setattr(bmg._lib, "Opts", make)
    B = bmg.Batch(9, [p[0] for p in probs], **kw)
    monkeypatch.undo()
    rhs = [p[1] for p in probs]
    counts = []
    for maxit in (0, 4):
        before = B.launch_count
        xs, _, _, _ = B.solve(rhs, tol=0.0, maxit=maxit)
        counts.append(B.launch_count - before)
    out = [x.clone() for x in xs], [B.history(k) for k in range(len(probs))]
    B.close()
    # (four iterations are one chunk, after which the done flags are gathered once more)
    return (counts[1] - counts[0] - 1) / 4, out


@pytest.mark.parametrize("precision,tail", [("fp32", 1), ("fp64", 1)])
def test_batched_halves_follow_the_restriction_option(bmg, monkeypatch, precision, tail):
    """BMG_FUSE_AUTO: the stages at 255 and 127 (FP64: 63) by halves; OFF: every step a launch of its own; ON: no
    halves either, so that one-pass stages take the pass that the option asks for.  Same bits."""
    probs = [problem(n) for n in ((255, 255, 127) if precision == "fp32" else (63, 63))]
    kw = dict(precision=precision, arith="fused")
    auto, a = batch_iteration(bmg, monkeypatch, probs, 0, **kw)
    off, b = batch_iteration(bmg, monkeypatch, probs, 1, **kw)
    on, c = batch_iteration(bmg, monkeypatch, probs, 2, **kw)
    # two launches a stage, the tail, then FP64 residual and norm, or FP32 update, residual and norm
    assert auto == (2 * 2 + tail + 3 if precision == "fp32" else 2 * 1 + tail + 2)
    assert off > auto and on > auto
    for x in (b, c):
        assert all(torch.equal(p, q) for p, q in zip(a[0], x[0])) and a[1] == x[1]


@pytest.mark.parametrize("precision,n,count,shared,halves", [
    ("fp64", 63, 9, False, 1), ("fp64", 63, 10, False, 0), ("fp32", 127, 130, False, 1), ("fp32", 255, 72, False, 2),
    ("fp32", 255, 74, False, 1), ("fp32", 255, 32, True, 2), ("fp32", 255, 33, True, 1), ("bf16", 511, 18, False, 3),
    ("bf16", 511, 19, False, 2), ("fp32", 511, 2, True, 2)])
def test_batched_halves_end_where_their_halos_cost_more(bmg, monkeypatch, precision, n, count, shared, halves):
    """On both sides of the lines that the rule draws; stages below the one named stay by halves."""
    coef, f = problem(n)
    h = bmg.Hierarchy(9, coef, precision=precision, arith="fused")
    B = bmg.Batch.from_hierarchy(h, count) if shared else bmg.Batch(9, [coef] * count, precision=precision, arith="fused")
    counts = []
    for maxit in (0, 4):
        before = B.launch_count
        B.solve([f] * count, tol=0.0, maxit=maxit)
        counts.append(B.launch_count - before)
    got, outer = (counts[1] - counts[0] - 1) / 4, 2 if precision == "fp64" else 3
    by_halves = 2 * halves + 1 + outer
    stages = {63: 1, 127: 1, 255: 2, 511: 3}[n]
    assert got == by_halves if halves == stages else got >= by_halves + 3
    B.close()
    h.close()


def solve_iteration(h, rhs):
    """Launches of one iteration of h."""
    counts = []
    for maxit in (0, 4):
        before = h.launch_count
        h.solve(rhs, tol=0.0, maxit=maxit)
        counts.append(h.launch_count - before)
    return (counts[1] - counts[0]) / 4


# levels by halves of a single problem: FP64 31 .. 511 over a tail from 15, FP32 and BF16 up to 1023 over a tail from
# 63 (the first level below it that is not BF16); with FP32 63 the whole cycle is the tail
@pytest.mark.parametrize("precision,n,halves", [("fp64", 31, 1), ("fp64", 63, 2), ("fp64", 511, 5), ("fp32", 63, 0),
                                                ("fp32", 127, 1), ("fp32", 1023, 4), ("bf16", 127, 2),
                                                ("bf16", 1023, 4)])
@pytest.mark.parametrize("kind", [5, 9])
def test_levels_by_halves(bmg, precision, n, halves, kind):
    coef, f = problem(n, kind)
    outer = 2 if precision == "fp64" else 3          # residual and norm; update, residual and norm
    h = bmg.Hierarchy(kind, coef, precision=precision, arith="fused")
    assert solve_iteration(h, f) == 2 * halves + 1 + outer
    h.close()
    h = bmg.Hierarchy(kind, coef, precision=precision, arith="fused", use_graph=False)
    assert solve_iteration(h, f) > 2 * halves + 1 + outer
    h.close()


@pytest.mark.parametrize("precision,n,halves", [("fp32", 127, 1), ("fp64", 255, 4)])
def test_levels_by_halves_in_flexible_cg(bmg, precision, n, halves):
    coef, f = problem(n)
    h = bmg.Hierarchy(9, coef, precision=precision, krylov="fcg")
    # z.q, its sum, direction, A p, its sums, update, norm
    assert solve_iteration(h, f) == 2 * halves + 1 + 7
    h.close()


@pytest.mark.parametrize("axes", ["x", "y", "xy"])
@pytest.mark.parametrize("n", [15, 255, 511])
def test_periodic_levels_by_halves(bmg, axes, n):
    kind, planes, f, px, py = periodic_problem(n, axes, seed=80 + n, kind=9)
    for krylov, outer in (("none", 1), ("fcg", 4)):   # residual; z.q, direction, A p, update (each with its sum)
        h = bmg.Hierarchy(kind, torch.from_numpy(planes).cuda(), periodic=axes, krylov=krylov)
        assert solve_iteration(h, torch.from_numpy(f).cuda()) == 2 * (h.num_levels - 1) + 1 + outer
        h.close()

"""Line relaxation of a hierarchy (factored lines, several lines to a CTA by the
number of lines) against the same V-cycle composed of the single-step entry
points, whose line kernels divide at every point: bit for bit at sizes on each
side of the lines-per-CTA rule, and with operators and right-hand sides scaled
so far that quotients overflow, underflow or become subnormal."""
import pytest
import torch

import workloads as w

pytestmark = pytest.mark.gpu


def composed_cycle(bmg, h, kind, f, axes, sweeps, level=0):
    """One V(sweeps, sweeps) cycle from zero on h's own operators."""
    A = h.stencil(level)
    k = kind if level == 0 else 9
    x = torch.zeros_like(f)
    if level == h.num_levels - 1:
        return bmg.coarse_solve(bmg.coarse_factor(A), f, x)

    def smooth():
        for _ in range(sweeps):
            for a in axes:
                bmg.relax_line(k, A, f, x, 1, axis=a)
    smooth()
    ci = h.interp(level)
    fc = bmg.resid_restrict(k, A, ci, x, f)
    fc[0], fc[-1], fc[:, 0], fc[:, -1] = 0.0, 0.0, 0.0, 0.0
    bmg.interp_correct(ci, composed_cycle(bmg, h, kind, fc, axes, sweeps, level + 1), x)
    smooth()
    return x


def check(bmg, kind, coef, f, smoother, axes, sweeps=1):
    h = bmg.Hierarchy(kind, coef, smoother=smoother, nu1=sweeps, nu2=sweeps)
    x, it, rr, ok = h.solve(f, tol=0.0, maxit=1)
    want = composed_cycle(bmg, h, kind, f, axes, sweeps)
    a, b = x[1:-1, 1:-1], want[1:-1, 1:-1]
    assert bool(((a == b) | (torch.isnan(a) & torch.isnan(b))).all())
    h.close()


@pytest.mark.parametrize("smoother,axes", [("line", "x"), ("yline", "y"), ("xyline", "xy")])
@pytest.mark.parametrize("n", [7, 255, 1023])
def test_line_cycle_is_the_composed_cycle(bmg, smoother, axes, n):
    coef = torch.from_numpy(w.fe9_from_cells(w.lognormal_cells(n, 2.0, 6.0, 70 + n))).cuda()
    check(bmg, 9, coef, torch.from_numpy(w.rhs_uniform(n, 71 + n)).cuda(), smoother, axes, sweeps=2)


@pytest.mark.parametrize("n", [4095, 8191])
def test_many_lines(bmg, n):
    coef = torch.from_numpy(w.anisotropic5(n, 1e-3)).cuda()[:3].contiguous()
    f = bmg.fill_uniform(n, 72)
    check(bmg, 5, coef, f, "xyline", "xy")


@pytest.mark.parametrize("op", [1.0, 2.0 ** -1000, 2.0 ** -500, 2.0 ** -201, 2.0 ** -199, 2.0 ** 199, 2.0 ** 600,
                                2.0 ** 960])
@pytest.mark.parametrize("rhs", [1.0, 2.0 ** -1040, 2.0 ** -450, 2.0 ** 480, 2.0 ** 1000])
def test_scaled_quotients(bmg, op, rhs):
    n = 63
    coef = torch.from_numpy(w.fe9_from_cells(w.lognormal_cells(n, 1.0, 6.0, 73)) * op).cuda()
    f = torch.from_numpy(w.rhs_uniform(n, 74) * rhs).cuda()
    if 2.0 ** -1000 < rhs < 2.0 ** 1000 and rhs / op < 2.0 ** 480:
        check(bmg, 9, coef, f, "xyline", "xy")
        return
    # a norm that underflows is a solved problem, one that overflows is refused
    h = bmg.Hierarchy(9, coef, smoother="xyline", nu1=1, nu2=1)
    if rhs <= 2.0 ** -1000:
        x, it, rr, ok = h.solve(f, tol=0.0, maxit=1)
        assert it == 0 and not bool(x.any())
    elif rhs >= 2.0 ** 1000:
        with pytest.raises(bmg.BmgError):
            h.solve(f, tol=0.0, maxit=1)
    h.close()

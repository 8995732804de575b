"""The work that users of the solver have it do, as cases to be measured.

A case is a dict of plain values.  `listed()` gives the named ones, `draw(rng)`
one more of the same ranges; `prepare` makes what a program holds before the
call (inputs on the GPU, and the hierarchy, batch or network it keeps), `run`
makes one pass through the public entry points, `work` says what the pass
cannot do without and `exact` what it computes, in 64 bits and in plain torch.

Families (the case's "do"):
  solve   one problem solved with a kept hierarchy (a time step, a Newton step
          with a frozen operator, one right-hand side after another)
  setup   the hierarchy built, one solve, the hierarchy released (the operator
          changes with every call)
  batch   many independent problems of uneven sizes solved together
  rhs     many right-hand sides of one operator
  train   one training step of the interpolation network on a batch of crops
  infer   the network's interpolation weights for one operator
"""
import math

import numpy as np
import torch

import paper_2502_05279_gb300 as bmg

DEV = "cuda"
F64 = torch.float64
SIDES = (63, 127, 255, 511, 1023)      # the sides that an uneven batch is made of
PARAMS = 18 * 64 + 64 + 64 * 64 + 64 + 64 * 4 + 4


# ---- the cases -----------------------------------------------------------------

def _solve(**kw):
    c = dict(do="solve", nx=127, ny=127, field="lognormal", strength=2.0, periodic="", precision="fp64",
             krylov="none", inner=1, arith="fused", smoother="auto", tol=1e-10)
    c.update(kw)
    return c


def listed():
    return [
        # the smallest solve: a 5-point Poisson problem with every option left alone
        _solve(name="poisson127-fp64", field="poisson", arith="rounded"),
        # a grid of no special size, every option left alone (embedded in the next 2^m - 1)
        _solve(name="rect300x200-fp64", nx=300, ny=200, strength=1.0, arith="rounded"),
        # an anisotropic operator, which needs x-line relaxation
        _solve(name="line511-fp64", nx=511, ny=511, field="aniso", strength=1e-3, smoother="line", arith="rounded"),
        # a new operator for every solve (coefficients that follow the solution)
        _solve(name="setup1023-fp32-fcg", do="setup", nx=1023, ny=1023, precision="fp32", krylov="fcg", inner=2),
        # a two-material problem with a contrast of 1e4: many accelerated FP32 cycles
        _solve(name="binary2047-fp32-fcg", nx=2047, ny=2047, field="binary", strength=1e4, precision="fp32",
               krylov="fcg", inner=2),
        # a large heterogeneous problem with BF16 stencils on the finest levels
        _solve(name="lognormal4095-bf16-fcg", nx=4095, ny=4095, precision="bf16", krylov="fcg", inner=2),
        # the largest grid, in FP64 throughout
        _solve(name="lognormal8191-fp64-fcg", nx=8191, ny=8191, krylov="fcg"),
        # a domain that is periodic along x
        _solve(name="periodic2048-fp64-fcg", nx=2048, ny=2047, periodic="x", krylov="fcg"),
        # forty independent problems of uneven sizes
        dict(name="batch40-fp32", do="batch", count=40, strength=1.0, precision="fp32", arith="fused", tol=1e-8),
        # sixteen right-hand sides of one operator
        dict(name="rhs16-1023-fp32", do="rhs", count=16, n=1023, strength=2.0, precision="fp32", arith="fused",
             tol=1e-10),
        # one optimizer step on the trainer's default batch of crops
        dict(name="train152-crop31", do="train", crops=152, n=31, vectors=4),
        # weights of a large operator from the trained network
        dict(name="infer2047", do="infer", n=2047, contrast=1e6),
    ]


def _log_int(rng, lo, hi):
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def _side(rng, lo, hi):
    """A size 2^m - 1 half of the time, else any size, log-uniform in lo .. hi."""
    n = _log_int(rng, lo, hi)
    if rng.random() < 0.5:
        m = 2 ** int(round(math.log2(n + 1))) - 1
        n = m if lo <= m <= hi else n
    return n


def draw(rng):
    kind = rng.choice(["solve", "solve", "solve", "line", "setup", "periodic", "batch", "rhs", "train", "infer"])
    arith = rng.choice(["rounded", "fused"])
    if kind in ("solve", "setup"):
        nx = _side(rng, 60, 2100 if kind == "solve" else 1100)
        ny = nx if rng.random() < 0.5 else max(40, int(nx * rng.uniform(0.4, 1.0)))
        precision = rng.choice(["fp64", "fp32", "bf16"])
        krylov = rng.choice(["none", "fcg"])
        field, strength = rng.choice([("poisson", 0.0), ("lognormal", 1.0), ("lognormal", 2.0), ("binary", 100.0)])
        return _solve(do=kind, nx=nx, ny=ny, field=field, strength=strength, precision=precision,
                      krylov="fcg" if field == "binary" else krylov, arith=arith,
                      inner=rng.choice([1, 2]) if precision != "fp64" else 1)
    if kind == "line":
        n = _side(rng, 60, 400)
        return _solve(nx=n, ny=n, field="aniso", strength=10.0 ** rng.uniform(-4, -2),
                      smoother=rng.choice(["line", "xyline"]), precision=rng.choice(["fp64", "fp32"]), arith=arith)
    if kind == "periodic":
        n = 2 ** rng.randint(6, 11) - 1
        axis = rng.choice(["x", "y"])
        return _solve(nx=n + (axis == "x"), ny=n + (axis == "y"), strength=rng.uniform(0.5, 2.0), periodic=axis,
                      krylov=rng.choice(["none", "fcg"]), arith=arith)
    if kind == "batch":
        return dict(do="batch", count=_log_int(rng, 4, 40), strength=rng.uniform(0.5, 1.5),
                    precision=rng.choice(["fp64", "fp32", "bf16"]), arith=arith, tol=1e-8)
    if kind == "rhs":
        n = 2 ** rng.randint(6, 10) - 1
        return dict(do="rhs", count=_log_int(rng, 2, 24), n=n, strength=rng.uniform(0.5, 2.0),
                    precision=rng.choice(["fp64", "fp32"]), arith=arith, tol=1e-10)
    if kind == "train":
        return dict(do="train", crops=_log_int(rng, 8, 304), n=rng.choice([15, 31]), vectors=rng.randint(1, 6))
    return dict(do="infer", n=2 ** rng.randint(7, 12) - 1, contrast=10.0 ** rng.uniform(2, 6))


# ---- inputs --------------------------------------------------------------------

def _rng(seed, stream):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed) * 1000 + stream)
    return g


def _gaussian(cells, std, g, corr=32.0):
    """A periodic Gaussian field of correlation length `corr` cells, sample std `std`."""
    w = torch.randn(cells, cells, generator=g, device=DEV, dtype=F64)
    k = 2.0 * math.pi * torch.fft.fftfreq(cells, device=DEV, dtype=F64)
    h = torch.exp(-0.25 * corr * corr * k * k)
    w = torch.fft.ifft2(torch.fft.fft2(w) * (h[:, None] * h[None, :])).real
    w = w - w.mean()
    return w * (std / w.std(correction=0))


def _blocks(cells, block, hi, g):
    nb = -(-cells // block)
    t = torch.where(torch.rand(nb, nb, generator=g, device=DEV, dtype=F64) < 0.5, hi, 1.0)
    return t.repeat_interleave(block, 0).repeat_interleave(block, 1)[:cells, :cells]


def _q1(k, px=False, py=False):
    """Planes O, W, S, SW, NW of the bilinear element stencil of -div(k grad u), k per cell (batch
    dimensions in front); the couplings to points outside the grid are zero."""
    if px:
        k = torch.cat([k, k[..., :, :1]], -1)
    if py:
        k = torch.cat([k, k[..., :1, :]], -2)
    ny, nx = k.shape[-2] - 1, k.shape[-1] - 1
    a, b, c, d = k[..., :ny, :nx], k[..., :ny, 1:], k[..., 1:, :nx], k[..., 1:, 1:]
    out = torch.zeros(*k.shape[:-2], 5, ny + 2, nx + 2, device=DEV, dtype=F64)
    v = out[..., 1:-1, 1:-1]
    v[..., 0, :, :] = (2.0 / 3.0) * (a + b + c + d)
    v[..., 1, :, :] = -(a + c) / 6.0
    v[..., 2, :, :] = -(a + b) / 6.0
    v[..., 3, :, :] = -a / 3.0
    v[..., 4, :, :] = -c / 3.0
    if not px:
        v[..., (1, 3, 4), :, 0] = 0.0
    if not py:
        v[..., (2, 3), 0, :] = 0.0
        v[..., 4, ny - 1, :] = 0.0
    return out


def _five(nx, ny, wx, wy):
    """Planes O, W, S of the 5-point operator -(wx u_xx + wy u_yy), unscaled."""
    out = torch.zeros(3, ny + 2, nx + 2, device=DEV, dtype=F64)
    out[0, 1:-1, 1:-1] = 2.0 * (wx + wy)
    out[1, 1:-1, 2:-1] = -wx
    out[2, 2:-1, 1:-1] = -wy
    return out


def _operator(case, seed):
    """(kind, planes) of a solve's operator."""
    nx, ny, g = case["nx"], case["ny"], _rng(seed, 1)
    if case["field"] == "poisson":
        return 5, _five(nx, ny, 1.0, 1.0)
    if case["field"] == "aniso":
        return 5, _five(nx, ny, 1.0, case["strength"])
    px, py = "x" in case["periodic"], "y" in case["periodic"]
    cells = max(nx + (not px), ny + (not py))
    if case["field"] == "binary":
        k = _blocks(cells, 16, case["strength"], g)
    else:
        k = torch.exp(_gaussian(cells, case["strength"], g))
    return 9, _q1(k[:ny + (not py), :nx + (not px)], px, py).contiguous()


def _rhs(nx, ny, g):
    f = torch.zeros(ny + 2, nx + 2, device=DEV, dtype=F64)
    f[1:-1, 1:-1] = 2.0 * torch.rand(ny, nx, generator=g, device=DEV, dtype=F64) - 1.0
    return f


def _hierarchy(case, kind, planes):
    return bmg.Hierarchy(kind, planes, precision=case["precision"], krylov=case["krylov"], inner_cycles=case["inner"],
                         arith=case["arith"], smoother=case["smoother"], periodic=case["periodic"])


def _batch_sides(count):
    return [SIDES[i % len(SIDES)] for i in range(count)]


def _batch_inputs(case, seed):
    planes, fs = [], []
    for i, n in enumerate(_batch_sides(case["count"])):
        planes.append(_q1(torch.exp(_gaussian(n + 1, case["strength"], _rng(seed, 10 + 2 * i)))))
        fs.append(_rhs(n, n, _rng(seed, 11 + 2 * i)))
    return planes, fs


def _rhs_inputs(case, seed):
    n = case["n"]
    planes = _q1(torch.exp(_gaussian(n + 1, case["strength"], _rng(seed, 1))))
    return planes, [_rhs(n, n, _rng(seed, 10 + i)) for i in range(case["count"])]


def _network(seed):
    """A parameter vector as training leaves it: scaled layers and a small output layer."""
    g = _rng(seed, 3)
    z = torch.randn(PARAMS, generator=g, device=DEV, dtype=torch.float32)
    z[:1152] *= math.sqrt(2.0 / 18)
    z[1152:1216] *= 0.05
    z[1216:5312] *= math.sqrt(2.0 / 64)
    z[5312:5376] *= 0.05
    z[5376:] *= 0.02
    return z


def _train_inputs(case, seed):
    """Crops of the high-contrast two-material family, tile-aligned, and error vectors."""
    C, n, K, g = case["crops"], case["n"], case["vectors"], _rng(seed, 4)
    nb = (n + 1) // 8
    k = torch.where(torch.rand(C, nb, nb, generator=g, device=DEV, dtype=F64) < 0.5, 1e6, 1.0)
    coefs = _q1(k.repeat_interleave(8, 1).repeat_interleave(8, 2)).contiguous()
    vecs = torch.zeros(C, K, n + 2, n + 2, device=DEV, dtype=F64)
    vecs[..., 1:-1, 1:-1] = 2.0 * torch.rand(C, K, n, n, generator=g, device=DEV, dtype=F64) - 1.0
    return coefs, vecs


def prepare(case, seed):
    do, state = case["do"], {"case": case}
    if do in ("solve", "setup"):
        kind, planes = _operator(case, seed)
        state.update(kind=kind, planes=planes, f=_rhs(case["nx"], case["ny"], _rng(seed, 2)))
        if do == "solve":
            state["h"] = _hierarchy(case, kind, planes)
    elif do == "batch":
        planes, fs = _batch_inputs(case, seed)
        state.update(fs=fs, batch=bmg.Batch(9, planes, precision=case["precision"], arith=case["arith"]))
    elif do == "rhs":
        planes, fs = _rhs_inputs(case, seed)
        h = bmg.Hierarchy(9, planes, precision=case["precision"], arith=case["arith"])
        state.update(fs=fs, h=h, batch=bmg.Batch.from_hierarchy(h, case["count"]))
    elif do == "train":
        coefs, vecs = _train_inputs(case, seed)
        net = bmg.Mlp(_network(seed).cpu().numpy())
        state.update(net=net, coefs=coefs, vecs=vecs, eref=net.twogrid(coefs, vecs)[2])
    else:
        n = case["n"]
        state.update(net=bmg.Mlp(_network(seed).cpu().numpy()),
                     planes=_q1(_blocks(n + 1, 8, case["contrast"], _rng(seed, 1))).contiguous())
    return state


# ---- one pass ------------------------------------------------------------------

def run(state):
    case = state["case"]
    do = case["do"]
    if do == "solve":
        x, iters, relres, _ = state["h"].solve(state["f"], tol=case["tol"])
        return {"x": x, "iters": iters}
    if do == "setup":
        h = _hierarchy(case, state["kind"], state["planes"])
        x, iters, relres, _ = h.solve(state["f"], tol=case["tol"])
        h.close()
        return {"x": x, "iters": iters}
    if do in ("batch", "rhs"):
        xs, iters, relres, _ = state["batch"].solve(state["fs"], tol=case["tol"])
        return {"xs": xs, "iters": np.array(iters)}
    if do == "train":
        loss, grad, energies = state["net"].twogrid(state["coefs"], state["vecs"], state["eref"])
        state["net"].adam(1e-4)
        return {"loss": loss, "grad": grad, "energies": energies}
    delta = state["net"].infer(state["planes"])
    return {"delta": delta, "weights": bmg.learned_interp(state["planes"], delta)}


# ---- what a pass cannot do without ---------------------------------------------

def work(case):
    """Each input read once and each output written once; flops of a solve: ten V(2,1) cycles
    (three sweeps, residual, restriction, interpolation: about 80 per point over all levels 4/3)."""
    do = case["do"]
    if do in ("solve", "setup"):
        pts = [(case["nx"] + 2) * (case["ny"] + 2)]
        planes = 3 if case["field"] in ("poisson", "aniso") else 5
    elif do == "batch":
        pts, planes = [(n + 2) ** 2 for n in _batch_sides(case["count"])], 5
    elif do == "rhs":
        pts, planes = [(case["n"] + 2) ** 2] * case["count"], 5 / case["count"]
    elif do == "train":
        C, n, K = case["crops"], case["n"], case["vectors"]
        m = ((n - 1) // 2) ** 2
        band = (n - 1) // 2 + 1
        return {"bytes": 8.0 * C * (5 + K) * (n + 2) ** 2 + 8.0 * C * K + 4.0 * PARAMS,
                "flops": C * (m * band * band + K * (m * 8 * band + 12 * 18 * n * n) + 3 * m * 11008.0)}
    else:
        nc = (case["n"] - 1) // 2
        return {"bytes": 40.0 * (case["n"] + 2) ** 2 + 16.0 * nc * nc + 64.0 * (nc + 2) ** 2 + 4.0 * PARAMS,
                "flops": nc * nc * (11008.0 + 60.0)}
    return {"bytes": 8.0 * (planes + 2) * sum(pts), "flops": 10 * 80 * 4 / 3 * float(sum(pts))}


# ---- the same in 64 bits, in plain torch ---------------------------------------

def _entries(planes, px=False):
    """The nine couplings a(p, p + (dx, dy)) of every interior point, as a dict over (dx, dy)."""
    p = planes.clone()
    if px:
        p[..., -1] = p[..., 1]
    if p.shape[-3] == 3:
        p = torch.cat([p, torch.zeros_like(p[..., :2, :, :])], -3)
    O, W, S, SW, NW = (p[..., i, :, :] for i in range(5))
    c = slice(1, -1)
    return {(0, 0): O[..., c, c], (-1, 0): W[..., c, c], (1, 0): W[..., c, 2:], (0, -1): S[..., c, c],
            (0, 1): S[..., 2:, c], (-1, -1): SW[..., c, c], (1, 1): SW[..., 2:, 2:], (-1, 1): NW[..., c, c],
            (1, -1): NW[..., :-2, 2:]}


def _direct(planes, fs, px=False):
    """A^-1 f for every f in fs by block elimination over the grid rows (periodic in x only)."""
    a = _entries(planes, px)
    ny, nx = a[(0, 0)].shape
    idx = torch.arange(nx, device=DEV)

    def block(j, dy):
        m = torch.zeros(nx, nx, device=DEV, dtype=F64)
        for dx in (-1, 0, 1):
            q = idx + dx
            ok = (q >= 0) & (q < nx) if not px else torch.ones_like(q, dtype=torch.bool)
            m[idx[ok], q[ok] % nx] += a[(dx, dy)][j][ok]
        return m

    f = torch.stack([x[1:-1, 1:-1] for x in fs], -1)       # ny, nx, right-hand sides
    y, inv = f.clone(), []
    for j in range(ny):
        d = block(j, 0)
        if j:
            low = block(j, -1)
            d = d - low @ inv[-1] @ block(j - 1, 1)
            y[j] = f[j] - low @ (inv[-1] @ y[j - 1])
        inv.append(torch.linalg.inv(d))
    x = torch.empty_like(y)
    for j in range(ny - 1, -1, -1):
        x[j] = inv[j] @ (y[j] - block(j, 1) @ x[j + 1] if j + 1 < ny else y[j])
    out = []
    for q in range(len(fs)):
        z = torch.zeros_like(fs[q])
        z[1:-1, 1:-1] = x[..., q]
        out.append(z)
    return out


def _mlp(theta, X):
    W1, b1, W2, b2 = theta[:1152].view(18, 64), theta[1152:1216], theta[1216:5312].view(64, 64), theta[5312:5376]
    W3, b3 = theta[5376:5632].view(64, 4), theta[5632:]
    h = torch.nn.functional.gelu(X @ W1 + b1)
    return torch.nn.functional.gelu(h @ W2 + b2) @ W3 + b3


def _features(a, nc):
    fx, fy = (a[(-1, 0)] + a[(1, 0)]) / a[(0, 0)], (a[(0, -1)] + a[(0, 1)]) / a[(0, 0)]
    cols = []
    for dy in (-1, 0, 1):
        for dx in (-1, 0, 1):
            s = (..., slice(1 + dy, 2 * nc + dy, 2), slice(1 + dx, 2 * nc + dx, 2))
            cols += [fx[s].flatten(-2), fy[s].flatten(-2)]
    return torch.stack(cols, -1)


def _weights(a, delta):
    """The eight weight planes (nc+2)^2 of logits delta (..., nc, nc, 4)."""
    nc = delta.shape[-2]
    n = 2 * nc + 1
    lead = delta.shape[:-3]
    dg = torch.nn.functional.pad(delta.movedim(-1, -3), (1, 1, 1, 1))
    o, e = slice(0, n, 2), slice(1, n - 1, 2)
    X, Y, Cn = (..., e, o), (..., o, e), (..., o, o)
    zero = torch.zeros(*lead, nc + 2, nc + 2, device=DEV, dtype=F64)

    def put(v, rows, cols):
        z = zero.clone()
        z[..., rows, cols] = v
        return z

    cw, ce = a[(-1, -1)][X] + a[(-1, 0)][X] + a[(-1, 1)][X], a[(1, -1)][X] + a[(1, 0)][X] + a[(1, 1)][X]
    sd = -(cw + ce) / (a[(0, -1)][X] + a[(0, 0)][X] + a[(0, 1)][X])
    u, v = cw * torch.exp(dg[..., 1, 1:nc + 1, 0:nc + 1]), ce * torch.exp(dg[..., 0, 1:nc + 1, 1:nc + 2])
    inner, wide = slice(1, nc + 1), slice(1, nc + 2)
    LL, LR = put(sd * u / (u + v), inner, wide), put(sd * v / (u + v), inner, wide)
    rs, rn = a[(-1, -1)][Y] + a[(0, -1)][Y] + a[(1, -1)][Y], a[(-1, 1)][Y] + a[(0, 1)][Y] + a[(1, 1)][Y]
    sd = -(rs + rn) / (a[(-1, 0)][Y] + a[(0, 0)][Y] + a[(1, 0)][Y])
    u, v = rs * torch.exp(dg[..., 3, 0:nc + 1, 1:nc + 1]), rn * torch.exp(dg[..., 2, 1:nc + 2, 1:nc + 1])
    LB, LA = put(sd * u / (u + v), wide, inner), put(sd * v / (u + v), wide, inner)
    B, W = slice(1, nc + 2), slice(0, nc + 1)
    q = {d: a[d][Cn] / a[(0, 0)][Cn] for d in a}
    SW = -(q[(-1, -1)] + q[(-1, 0)] * LB[..., B, W] + q[(0, -1)] * LL[..., W, B])
    SE = -(q[(1, -1)] + q[(1, 0)] * LB[..., B, B] + q[(0, -1)] * LR[..., W, B])
    NW = -(q[(-1, 1)] + q[(-1, 0)] * LA[..., B, W] + q[(0, 1)] * LL[..., B, B])
    NE = -(q[(1, 1)] + q[(1, 0)] * LA[..., B, B] + q[(0, 1)] * LR[..., B, B])
    return torch.stack([put(t, B, B) for t in (SW, SE, NW, NE)] + [LL, LR, LB, LA], -3)


def _dense(a):
    """Dense matrices (..., n^2, n^2) of the couplings a."""
    n = a[(0, 0)].shape[-1]
    lead = a[(0, 0)].shape[:-2]
    A = torch.zeros(*lead, n, n, n, n, device=DEV, dtype=F64)
    j, i = torch.meshgrid(torch.arange(n, device=DEV), torch.arange(n, device=DEV), indexing="ij")
    for (dx, dy), v in a.items():
        ok = (j + dy >= 0) & (j + dy < n) & (i + dx >= 0) & (i + dx < n)
        A[..., j[ok], i[ok], j[ok] + dy, i[ok] + dx] = v[..., ok]
    return A.reshape(*lead, n * n, n * n)


def _prolongation(w):
    """Dense P (..., n^2, nc^2) of the weight planes w."""
    nc = w.shape[-1] - 2
    n = 2 * nc + 1
    P = torch.zeros(*w.shape[:-3], n + 2, n + 2, nc + 2, nc + 2, device=DEV, dtype=F64)
    jc, ic = torch.meshgrid(torch.arange(1, nc + 2, device=DEV), torch.arange(1, nc + 2, device=DEV), indexing="ij")
    SW, SE, NW, NE, LL, LR, LB, LA = (w[..., k, 1:, 1:] for k in range(8))
    P[..., 2 * jc, 2 * ic, jc, ic] = torch.ones_like(SW)
    for v, dj, di in ((LL, 0, -1), (LR, 0, 0)):
        P[..., 2 * jc, 2 * ic - 1, jc + dj, ic + di] = v
    for v, dj, di in ((LB, -1, 0), (LA, 0, 0)):
        P[..., 2 * jc - 1, 2 * ic, jc + dj, ic + di] = v
    for v, dj, di in ((SW, -1, -1), (SE, -1, 0), (NW, 0, -1), (NE, 0, 0)):
        P[..., 2 * jc - 1, 2 * ic - 1, jc + dj, ic + di] = v
    return P[..., 1:-1, 1:-1, 1:-1, 1:-1].reshape(*w.shape[:-3], n * n, nc * nc)


def _energies(A, w, vecs):
    """||S (I - P Ac^-1 P^T A) S^2 e||_A^2 of every error vector (crops, K, n^2)."""
    n = int(round(math.sqrt(A.shape[-1])))
    P, e = _prolongation(w), vecs.transpose(-1, -2)
    j, i = torch.meshgrid(torch.arange(1, n + 1, device=DEV), torch.arange(1, n + 1, device=DEV), indexing="ij")
    D = torch.diagonal(A, dim1=-2, dim2=-1)[..., None]

    def sweep(x):
        for pi, pj in ((1, 1), (0, 1), (1, 0), (0, 0)):
            on = ((i % 2 == pi) & (j % 2 == pj)).reshape(-1, 1)
            x = torch.where(on, x - (A @ x) / D, x)
        return x

    e = sweep(sweep(e))
    Pt = P.transpose(-1, -2)
    e = e - P @ torch.linalg.solve(Pt @ A @ P, Pt @ (A @ e))
    e = sweep(e)
    return (e * (A @ e)).sum(-2)


def _train_exact(case, seed):
    coefs, vecs = _train_inputs(case, seed)
    C, K, n = case["crops"], case["vectors"], case["n"]
    nc, flat = (n - 1) // 2, vecs[..., 1:-1, 1:-1].reshape(C, K, n * n)
    theta = _network(seed).double().requires_grad_()
    loss, grad, got = 0.0, torch.zeros_like(theta), []
    for c in range(0, C, 16):
        a = _entries(coefs[c:c + 16])
        A, m = _dense(a), a[(0, 0)].shape[0]
        with torch.no_grad():
            ref = _energies(A, _weights(a, torch.zeros(m, nc, nc, 4, device=DEV, dtype=F64)), flat[c:c + 16])
        E = _energies(A, _weights(a, _mlp(theta, _features(a, nc)).view(m, nc, nc, 4)), flat[c:c + 16])
        part = (E / ref).sum() / (C * K)
        grad += torch.autograd.grad(part, theta)[0]
        loss += float(part.detach())
        got.append(E.detach())
    return {"loss": loss, "grad": grad, "energies": torch.cat(got)}


def exact(case, seed):
    do = case["do"]
    if do in ("solve", "setup"):
        if max(case["nx"], case["ny"]) > 513 or "y" in case["periodic"]:
            return None
        _, planes = _operator(case, seed)
        f = _rhs(case["nx"], case["ny"], _rng(seed, 2))
        return {"x": _direct(planes, [f], "x" in case["periodic"])[0], "iters": None}
    if do == "batch":
        planes, fs = _batch_inputs(case, seed)
        return {"xs": [_direct(p, [f])[0] if f.shape[0] < 140 else None for p, f in zip(planes, fs)], "iters": None}
    if do == "rhs":
        if case["n"] > 511:
            return None
        planes, fs = _rhs_inputs(case, seed)
        return {"xs": _direct(planes, fs), "iters": None}
    if do == "train":
        return _train_exact(case, seed)
    n = case["n"]
    nc = (n - 1) // 2
    a = _entries(_q1(_blocks(n + 1, 8, case["contrast"], _rng(seed, 1))))
    delta = _mlp(_network(seed).double(), _features(a, nc))
    return {"delta": delta, "weights": _weights(a, delta.view(nc, nc, 4))}

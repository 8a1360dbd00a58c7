"""What a user of this library runs most: the Galerkin operator (hom_matvec) in its three
arithmetics, whole bound computations (hom_bounds, hom_bounds_batched) and the warm-start
network (one training step, one prediction), each through the Python binding of the C ABI.

    listed()            the cases, plain dicts
    draw(rng)           one more case of the same ranges
    prepare(case, seed) inputs, context and workspace of one case
    run(state)          one pass
    work(case)          bytes and operations one pass cannot do without
    exact(case, seed)   what run returns, from plain torch in 64 bits (None where it has no such value)
"""
import math

import numpy as np
import torch

import microstructures as ms

DEV = "cuda"
PREC = {"fp64": 0, "mixed": 1, "fp32": 2, "ff": 3}
REAL = {"fp64": torch.float64, "fp32": torch.float32, "ff": torch.float64}
FIELD = {"fp64": torch.complex128, "fp32": torch.complex64, "ff": torch.complex128}


def listed():
    return [
        # the 2D square cell of the smallest configuration: three short launches and the host path
        {"name": "op2d_fp64_n23", "kind": "op", "d": 2, "nx": 23, "ny": 23, "nz": 1, "prec": "fp64", "side": 0, "aniso": False},
        # the largest 2D grid of the batched configuration, anisotropic phases, dual side
        {"name": "op2d_fp32_n203_aniso", "kind": "op", "d": 2, "nx": 203, "ny": 203, "nz": 1, "prec": "fp32", "side": 1, "aniso": True},
        # the operator of the 3D cube configuration, plain FP64 CG
        {"name": "op3d_fp64_n41", "kind": "op", "d": 3, "nx": 41, "ny": 41, "nz": 41, "prec": "fp64", "side": 0, "aniso": False},
        # the inner operator of the largest configuration (16 balls, double grid 225^3)
        {"name": "op3d_fp32_n113", "kind": "op", "d": 3, "nx": 113, "ny": 113, "nz": 113, "prec": "fp32", "side": 0, "aniso": False},
        # a box-shaped cell: another resolution on every axis, anisotropic phases, dual side
        {"name": "op3d_fp32_ragged_aniso", "kind": "op", "d": 3, "nx": 41, "ny": 33, "nz": 53, "prec": "fp32", "side": 1, "aniso": True},
        # the refinement residual's float-float operator
        {"name": "op3d_ff_n63", "kind": "op", "d": 3, "nx": 63, "ny": 63, "nz": 63, "prec": "ff", "side": 0, "aniso": False},
        # the smallest configuration as a whole: both bounds of the square cell in FP64 to 1e-8
        {"name": "bounds2d_fp64_n23", "kind": "bounds", "d": 2, "n": 23, "prec": "fp64", "tol": 1e-8, "contrast": 10.0},
        # 16 balls at contrast 1000 on an ordinary 3D grid, mixed precision
        {"name": "bounds3d_mixed_n51", "kind": "bounds", "d": 3, "n": 51, "prec": "mixed", "tol": 1e-6, "contrast": 1000.0},
        # the same cell on the largest configuration's grid
        {"name": "bounds3d_mixed_n113", "kind": "bounds", "d": 3, "n": 113, "prec": "mixed", "tol": 1e-6, "contrast": 1000.0},
        # random-rectangle cells with N from {23, 63, 113, 203} in one launch
        {"name": "batch2d_mixed_64", "kind": "batch", "cells": 64, "n": 0, "prec": "mixed", "tol": 1e-4},
        # one Adam step of the 2D warm-start network, its training batch
        {"name": "net_train_2d_n63", "kind": "net", "d": 2, "n": 63, "batch": 32, "width": 32, "modes": 12, "layers": 4, "proj": 128, "train": True},
        # prediction of the 3D warm-start network on its training grid
        {"name": "net_forward_3d_n41", "kind": "net", "d": 3, "n": 41, "batch": 8, "width": 24, "modes": 8, "layers": 4, "proj": 64, "train": False},
    ]


def _odd(rng, lo, hi):
    """An odd integer, spread over the logarithm of [lo, hi]."""
    n = int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))
    return min(hi, max(lo, n | 1))


def draw(rng):
    kind = rng.choice(["op", "op", "op", "op", "op", "op", "bounds", "bounds", "batch", "net", "net"])
    if kind == "op":
        d = rng.choice([2, 3, 3])
        lo, hi = (15, 203) if d == 2 else (11, 113)
        n = [_odd(rng, lo, hi)] * 3
        if rng.random() < 0.3:
            n = [_odd(rng, lo, hi) for _ in range(3)]
        return {"kind": "op", "d": d, "nx": n[0], "ny": n[1], "nz": n[2] if d == 3 else 1,
                "prec": rng.choice(["fp64", "fp32", "fp32", "ff"]), "side": rng.randrange(2), "aniso": rng.random() < 0.3}
    if kind == "bounds":
        d = rng.choice([2, 3, 3])
        prec = rng.choice(["fp64", "mixed", "mixed"])
        hi = 113 if d == 2 else (33 if prec == "fp64" else 81)
        return {"kind": "bounds", "d": d, "n": _odd(rng, 15, hi), "prec": prec, "tol": 1e-8 if prec == "fp64" else 1e-6,
                "contrast": round(10.0 ** rng.uniform(1.0, 3.0), 2)}
    if kind == "batch":
        return {"kind": "batch", "cells": rng.randrange(12, 65), "n": rng.choice([0, _odd(rng, 23, 113)]), "prec": "mixed",
                "tol": 1e-4}
    d = rng.choice([2, 3])
    n = _odd(rng, 31, 81) if d == 2 else _odd(rng, 21, 41)
    return {"kind": "net", "d": d, "n": n, "batch": rng.randrange(1, 33) if d == 2 else rng.randrange(1, 9),
            "width": rng.choice([24, 32]), "modes": rng.randrange(8, 13) if d == 2 else rng.randrange(4, 9), "layers": 4,
            "proj": rng.choice([64, 128]), "train": rng.random() < 0.5}


# ---------------------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------------------
def _spd(rng, d):
    q, _ = np.linalg.qr(rng.normal(size=(d, d)))
    return q @ np.diag(10.0 ** rng.uniform(-1, 1, size=d)) @ q.T


def _op_problem(c, seed):
    """One box in each half of the cell (and a ball in 3D), contrast 10 to 1000."""
    rng = np.random.default_rng([17, seed])
    d, N = c["d"], (c["nx"], c["ny"], c["nz"])[:c["d"]]
    Y = np.array([1.0, 0.9, 1.1][:d]) if c["aniso"] else np.ones(d)
    phase = (lambda: _spd(rng, d)) if c["aniso"] else (lambda: float(10.0 ** rng.uniform(1, 3)))
    shift = rng.uniform(-0.05, 0.05, size=d)
    left = np.array([-0.25] + [0.0] * (d - 1))
    incl = [ms.box((left + shift) * Y, rng.uniform(0.2, 0.38, size=d) * Y, phase(), d),
            ms.ball((-left + shift) * Y, float(rng.uniform(0.1, 0.18)), phase(), d)]
    return ms.make_problem(d, N, Y, _spd(rng, d) if c["aniso"] else 1.0, incl)


def _bounds_problem(c, seed):
    """2D: the centred square; 3D: 16 equal balls (fewer on the coarsest grids), seeded."""
    rng = np.random.default_rng([23, seed])
    if c["d"] == 2:
        return ms.square_inclusion_2d(N=c["n"], side=float(rng.uniform(0.5, 0.7)), a_incl=c["contrast"] * float(rng.uniform(0.9, 1.1)))
    return ms.random_spheres_3d(int(seed), N=c["n"], contrast=c["contrast"])


def _freq(n):
    return torch.fft.fftfreq(n, 1.0 / n, device=DEV, dtype=torch.float64)


def _double_grid_coef(p, side):
    """The coefficient of one side on the grid 2N - 1, [q, (z,) y, x]: closed-form Fourier
    coefficients of the boxes and balls, summed by an inverse transform."""
    d = p.d
    M = [2 * int(n) - 1 for n in p.N]
    xs = [_freq(M[a]) / float(p.Y[a]) for a in range(d)]
    xs[0] = torch.arange((M[0] + 1) // 2, device=DEV, dtype=torch.float64) / float(p.Y[0])
    shape = [[1] * d for _ in range(d)]
    for a in range(d):
        shape[a][d - 1 - a] = -1
    xi = [xs[a].reshape(shape[a]) for a in range(d)]
    A0 = np.linalg.inv(p.A0) if side else p.A0
    pairs = [(0, 0), (1, 1), (0, 1)] if d == 2 else [(0, 0), (1, 1), (2, 2), (1, 2), (0, 2), (0, 1)]
    pairs = pairs[:1] if p.is_isotropic() else pairs
    full = [1] * d
    for a in range(d):
        full[d - 1 - a] = xs[a].numel()
    hat = torch.zeros([len(pairs)] + full, dtype=torch.complex128, device=DEV)
    vol = float(np.prod(p.Y))
    for inc in p.inclusions:
        dA = (np.linalg.inv(inc.A) if side else inc.A) - A0
        phase = sum(xi[a] * float(inc.center[a]) for a in range(d))
        if inc.shape == ms.BOX:
            f = torch.ones(full, dtype=torch.float64, device=DEV)
            for a in range(d):
                f = f * float(inc.size[a]) * torch.sinc(xi[a] * float(inc.size[a]))
        else:
            r = float(inc.size[0])
            q = 2 * math.pi * r * torch.sqrt(sum(x * x for x in xi))
            s = torch.where(q > 1e-3, q, torch.ones_like(q))
            if d == 3:
                f = 4 * math.pi * r ** 3 * torch.where(q > 1e-3, (torch.sin(s) - s * torch.cos(s)) / s ** 3, 1 / 3 - q * q / 30)
            else:
                f = 2 * math.pi * r * r * torch.where(q > 1e-3, torch.special.bessel_j1(s) / s, 0.5 - q * q / 16)
        g = torch.polar(f / vol, -2 * math.pi * phase.expand(full).contiguous())
        for i, (a, b) in enumerate(pairs):
            hat[i] += float(dA[a, b]) * g
    for i, (a, b) in enumerate(pairs):
        hat[i].view(-1)[0] += float(A0[a, b])
    return torch.fft.irfftn(hat, s=M[::-1], dim=list(range(1, d + 1)), norm="forward")


def _random_fields(N, count, seed, dtype):
    """Half spectra [count, (z,) y, kx] of random real fields on the N grid."""
    g = torch.Generator(device=DEV).manual_seed(int(seed))
    v = torch.randn([count] + [int(n) for n in N[::-1]], generator=g, device=DEV, dtype=torch.float64)
    return torch.fft.rfftn(v, dim=list(range(1, len(N) + 1)), norm="forward").to(dtype)


def _op_inputs(c, seed):
    p = _op_problem(c, seed)
    a = _double_grid_coef(p, c["side"])
    if c["prec"] == "ff":   # pairs of floats, high and low part
        hi = a.float()
        coef = torch.stack([hi, (a - hi.double()).float()], dim=-1).contiguous()
    else:
        coef = a.to(REAL[c["prec"]]).contiguous()
    u = _random_fields([int(n) for n in p.N], c["d"] * c["d"], seed, FIELD[c["prec"]])
    return p, coef, u.reshape([c["d"], c["d"]] + list(u.shape[1:])).contiguous()


def _net_sizes(c):
    d, n, w, k = c["d"], c["n"], c["width"], c["modes"]
    return d, n, w, k, (2 * k) ** (d - 1) * k, 2 * d * d


def _net_inputs(c, seed):
    """Parameters of a network in training, features and targets of a batch of cells."""
    d, n, w, k, m, out = _net_sizes(c)
    g = torch.Generator(device=DEV).manual_seed(int(seed))

    def rnd(size, scale):
        return (torch.randn(size, generator=g, device=DEV) * scale).reshape(-1)
    parts = [rnd(w, 1.0), rnd(w, 0.1)]
    for _ in range(c["layers"]):
        parts += [rnd(2 * m * w * w, 1.0 / w), rnd(w * w, w ** -0.5), rnd(w, 0.1)]
    parts += [rnd(w * c["proj"], w ** -0.5), rnd(c["proj"], 0.1), rnd(c["proj"] * out, c["proj"] ** -0.5), rnd(out, 0.1)]
    params = torch.cat(parts)
    x = (torch.randn([c["batch"]] + [n] * d + [1], generator=g, device=DEV) > 0.5).float()
    x = x * (torch.rand([c["batch"]] + [1] * (d + 1), generator=g, device=DEV) * 5 / 3 - 2 / 3)
    t = torch.randn([c["batch"]] + [n] * d + [out], generator=g, device=DEV)
    mom = rnd(params.numel(), 1e-4)
    var = rnd(params.numel(), 1e-4) ** 2 + 1e-9
    return params, x, t, mom, var


def prepare(case, seed):
    import paper_1404_3614_gb300 as hb
    bd = hb.binding
    s = {"case": case, "hb": hb, "stream": torch.cuda.current_stream().cuda_stream}
    if case["kind"] == "op":
        p, coef, u = _op_inputs(case, seed)
        ctx = hb.hom_create(0)
        n = bd.hom_step_workspace_size(ctx, p, case["d"])
        s.update(p=p, coef=coef, u=u, out=torch.empty_like(u), ws=torch.empty(n, dtype=torch.uint8, device=DEV), ctx=_Context(hb, ctx))
    elif case["kind"] == "bounds":
        s.update(p=_bounds_problem(case, seed), solver=hb.Bounds(0))
    elif case["kind"] == "batch":
        cells = [ms.random_rectangles_2d(1000 * (int(seed) % 100000) + i, N=case["n"] or None) for i in range(case["cells"])]
        s.update(cells=cells, solver=hb.Bounds(0))
    else:
        d, n, w, k, m, out = _net_sizes(case)
        params, x, t, mom, var = _net_inputs(case, seed)
        ctx = hb.hom_create(0)
        cfg = bd.net_config(n, 1, w, k, case["layers"], case["proj"], out, d)
        n_params, nb = bd.hom_net_sizes(ctx, cfg, case["batch"])
        assert n_params == params.numel()
        s.update(cfg=cfg, params=params, x=x, t=t, m=mom, v=var, grad=torch.empty_like(params), loss=torch.zeros(1, device=DEV),
                 out=torch.empty_like(t), ws=torch.empty(nb, dtype=torch.uint8, device=DEV), ctx=_Context(hb, ctx))
    return s


class _Context:
    """A library context, destroyed with the state that holds it."""

    def __init__(self, hb, handle):
        self.hb, self.handle = hb, handle

    def __del__(self):
        try:
            self.hb.hom_destroy(self.handle)
        except Exception:
            pass


# ---------------------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------------------
def run(s):
    c, bd = s["case"], s["hb"].binding
    if c["kind"] == "op":
        bd.hom_matvec(s["ctx"].handle, s["p"], c["side"], PREC[c["prec"]], 1, c["d"], s["coef"].data_ptr(), s["u"].data_ptr(),
                      s["out"].data_ptr(), s["ws"].data_ptr(), s["ws"].numel(), s["stream"])
        return s["out"]
    if c["kind"] == "bounds":
        r = s["solver"](s["p"], precision=PREC[c["prec"]], tol=c["tol"])
        return {k: r[k] for k in ("upper", "lower", "mean", "D")}
    if c["kind"] == "batch":
        r = s["solver"].batched(s["cells"], precision=PREC[c["prec"]], tol=c["tol"])
        return {k: r[k] for k in ("upper", "lower")}
    if c["train"]:
        bd.hom_net_train_step(s["ctx"].handle, s["cfg"], s["params"].data_ptr(), s["m"].data_ptr(), s["v"].data_ptr(),
                              s["grad"].data_ptr(), 100, 2e-3, c["batch"], s["x"].data_ptr(), s["t"].data_ptr(),
                              s["loss"].data_ptr(), s["ws"].data_ptr(), s["ws"].numel(), s["stream"])
        return {k: s[k] for k in ("params", "m", "v", "grad", "loss")}
    bd.hom_net_forward(s["ctx"].handle, s["cfg"], s["params"].data_ptr(), c["batch"], s["x"].data_ptr(), s["out"].data_ptr(),
                       s["ws"].data_ptr(), s["ws"].numel(), s["stream"])
    return s["out"]


# ---------------------------------------------------------------------------------------
# bytes and operations of one pass
# ---------------------------------------------------------------------------------------
def _op_work(d, n, ncomp, fields, elem):
    """One operator application on `fields` components: fields in and out, the coefficient once;
    transforms at 5 M log2 M per complex pencil (half for a real row), both ways."""
    M = [2 * v - 1 for v in n]
    nh = (n[0] + 1) // 2

    def fft(m):
        return 5.0 * m * math.log2(m)
    f = 0.5 * fft(M[0]) * M[1] * (M[2] if d == 3 else 1) + nh * (M[2] if d == 3 else 1) * fft(M[1])
    if d == 3:
        f += nh * n[1] * fft(M[2])
    grid = M[0] * M[1] * (M[2] if d == 3 else 1)
    field = nh * n[1] * (n[2] if d == 3 else 1)
    return {"bytes": elem * (2 * fields * field) + elem / 2 * ncomp * grid,
            "flops": fields * (2 * f + 2 * grid * (1 if ncomp == 1 else d))}


def work(c):
    if c["kind"] == "op":
        d = c["d"]
        return _op_work(d, (c["nx"], c["ny"], c["nz"]), (d * (d + 1) // 2) if c["aniso"] else 1, d * d,
                        8 if c["prec"] == "fp32" else 16)
    if c["kind"] == "bounds":
        # CG steps at the usual rate for this contrast, the dual side half as many
        d, steps = c["d"], 1.5 * 0.5 * math.sqrt(c["contrast"]) * math.log(2 / c["tol"])
        w = _op_work(d, (c["n"],) * 3, 1, d * d, 8 if c["prec"] == "mixed" else 16)
        return {k: steps * v for k, v in w.items()}
    if c["kind"] == "batch":
        w = [_op_work(2, (n,) * 3, 1, 4, 8) for n in ([c["n"]] if c["n"] else [23, 63, 113, 203])]
        return {k: 1.5 * 60 * c["cells"] * sum(v[k] for v in w) / len(w) for k in ("bytes", "flops")}
    d, n, w, k, m, out = _net_sizes(c)
    pts = c["batch"] * n ** d
    row = n ** (d - 1) * c["batch"]
    spec = 4.0 * row * k * n * w + 8.0 * row * k * 2 * k * w * (1 if d == 2 else 1 + 2 * k / n)
    f = c["layers"] * (2 * spec + 8.0 * c["batch"] * m * w * w + 2.0 * pts * w * w) + 2.0 * pts * (w + w * c["proj"] + c["proj"] * out)
    params = w + w + c["layers"] * (2 * m * w * w + w * w + w) + w * c["proj"] + c["proj"] + c["proj"] * out + out
    if c["train"]:
        return {"bytes": 4.0 * (pts * (1 + out) + 7 * params), "flops": 3 * f}
    return {"bytes": 4.0 * (pts * (1 + out) + params), "flops": f}


# ---------------------------------------------------------------------------------------
# the same in 64 bits, plain torch
# ---------------------------------------------------------------------------------------
class _Operator:
    """Gamma P_N F_M (A_M / |M|) F_M^-1 Pad on half spectra [..., d, (z,) y, kx]."""

    def __init__(self, p, side, coef, project=True):
        self.d, self.side, self.coef, self.project = p.d, side, coef, project
        self.N = [int(n) for n in p.N]
        self.M = [int(v) for v in coef.shape[:0:-1]]
        d, nh = p.d, (self.N[0] + 1) // 2
        idx = [torch.arange(nh, device=DEV)]
        for a in range(1, d):
            k = torch.round(_freq(self.N[a])).long()
            idx.append(torch.where(k < 0, k + self.M[a], k))
        self.at = tuple(i.reshape([-1 if q == d - 1 - a else 1 for q in range(d)]) for a, i in reversed(list(enumerate(idx))))
        ks = [torch.arange(nh, device=DEV, dtype=torch.float64)] + [_freq(self.N[a]) for a in range(1, d)]
        self.xi = [(ks[a] / float(p.Y[a])).reshape([-1 if q == d - 1 - a else 1 for q in range(d)]) for a in range(d)]
        n2 = sum(x * x for x in self.xi)
        self.inv = torch.where(n2 > 0, 1 / torch.where(n2 > 0, n2, torch.ones_like(n2)), torch.zeros_like(n2))
        self.nonzero = (n2 > 0).double()

    def gamma(self, v):
        dot = sum(self.xi[c] * v[c] for c in range(self.d)) * self.inv
        g = torch.stack([self.xi[c] * dot for c in range(self.d)])
        return g if self.side == 0 else (v - g) * self.nonzero

    def __call__(self, u):
        """One field [d, (z,) y, kx]."""
        d = self.d
        full = torch.zeros([d] + self.M[:0:-1] + [(self.M[0] + 1) // 2], dtype=torch.complex128, device=DEV)
        full[(slice(None),) + self.at] = u.to(torch.complex128)
        dims = list(range(1, d + 1))
        x = torch.fft.irfftn(full, s=self.M[::-1], dim=dims, norm="forward")
        a = self.coef
        if a.shape[0] == 1:
            x = a * x
        else:
            o = {2: [[0, 2], [2, 1]], 3: [[0, 5, 4], [5, 1, 3], [4, 3, 2]]}[d]
            x = torch.stack([sum(a[o[i][j]] * x[j] for j in range(d)) for i in range(d)])
        v = torch.fft.rfftn(x, dim=dims, norm="forward")[(slice(None),) + self.at]
        return self.gamma(v) if self.project else v


def _energy_matrix(p, side, tol):
    """W[a, b] = a(e_b + x_b, e_a + x_a) of the CG minimisers of one side."""
    d = p.d
    coef = _double_grid_coef(p, side)
    C, raw = _Operator(p, side, coef), _Operator(p, side, coef, project=False)
    nh = (int(p.N[0]) + 1) // 2
    wt = torch.full([nh], 2.0, dtype=torch.float64, device=DEV)
    wt[0] = 1.0

    def dot(x, y):
        return float((wt * (x.conj() * y).real).sum())
    shape = [d] + [int(n) for n in p.N[:0:-1]] + [nh]
    us, W = [], np.zeros((d, d))
    for r in range(d):
        e = torch.zeros(shape, dtype=torch.complex128, device=DEV)
        e[r].view(-1)[0] = 1.0
        x = torch.zeros_like(e)
        res = -C(e)
        q, rr = res.clone(), dot(res, res)
        for _ in range(4000):
            if rr <= tol * tol:
                break
            Cq = C(q)
            al = rr / dot(q, Cq)
            x += al * q
            res = res - al * Cq
            new = dot(res, res)
            q, rr = res + (new / rr) * q, new
        us.append(e + C.gamma(x))
    for b in range(d):
        Au = raw(us[b])
        for a in range(d):
            W[a, b] = dot(us[a], Au)
    return 0.5 * (W + W.T)


def _net(c, params, x):
    d, n, w, k, m, out = _net_sizes(c)
    at = 0

    def take(*shape):
        nonlocal at
        size = int(np.prod(shape))
        v = params[at:at + size].reshape(shape)
        at += size
        return v

    def gelu(z):
        return 0.5 * z * (1 + torch.erf(z / math.sqrt(2.0)))
    dims = list(range(1, d + 1))
    ks = torch.cat([torch.arange(k), torch.arange(n - k, n)]).to(DEV)
    kept = tuple(i.reshape([-1 if q == a else 1 for q in range(d)]) for a, i in enumerate([ks] * (d - 1) + [torch.arange(k, device=DEV)]))
    v = x @ take(1, w) + take(w)
    for layer in range(c["layers"]):
        R = take(2, *([2 * k] * (d - 1) + [k]), w, w)
        y = torch.fft.fftn(v, dim=dims)[(slice(None),) + kept]
        y = torch.einsum("b...i,...ij->b...j", y, torch.complex(R[0], R[1]))
        wt = torch.full([k, 1], 2.0, dtype=torch.float64, device=DEV)
        wt[0] = 1.0
        z = torch.zeros([x.shape[0]] + [n] * d + [w], dtype=torch.complex128, device=DEV)
        z = z.index_put((torch.arange(x.shape[0], device=DEV).reshape([-1] + [1] * d),) + tuple(i.unsqueeze(0) for i in kept), y * wt)
        v2 = torch.fft.ifftn(z, dim=dims).real + v @ take(w, w) + take(w)
        v = gelu(v2) if layer + 1 < c["layers"] else v2
    v = gelu(v @ take(w, c["proj"]) + take(c["proj"]))
    return v @ take(c["proj"], out) + take(out)


def exact(case, seed):
    c = case
    if c["kind"] == "op":
        p, coef, u = _op_inputs(c, seed)
        a = (coef[..., 0].double() + coef[..., 1].double()) if c["prec"] == "ff" else coef.double()
        C = _Operator(p, c["side"], a)
        return torch.stack([C(v) for v in u])
    if c["kind"] == "bounds":
        if c["d"] == 3 and c["n"] > 51:   # some thousand transforms of a large grid
            return None
        p = _bounds_problem(c, seed)
        up = _energy_matrix(p, 0, 1e-11)
        lo = np.linalg.inv(_energy_matrix(p, 1, 1e-11))
        return {"upper": up, "lower": lo, "mean": 0.5 * (up + lo), "D": 0.5 * (up - lo)}
    if c["kind"] == "batch":
        return None
    params, x, t, mom, var = (v.double() for v in _net_inputs(c, seed))
    if not c["train"]:
        with torch.no_grad():
            return _net(c, params, x)
    params.requires_grad_(True)
    loss = ((_net(c, params, x) - t) ** 2).mean()
    grad, = torch.autograd.grad(loss, params)
    b1, b2 = 0.9, 0.999
    mom, var = b1 * mom + (1 - b1) * grad, b2 * var + (1 - b2) * grad ** 2
    new = params.detach() - 2e-3 * (mom / (1 - b1 ** 100)) / (torch.sqrt(var / (1 - b2 ** 100)) + 1e-8)
    return {"params": new, "m": mom, "v": var, "grad": grad, "loss": loss.detach().reshape(1)}

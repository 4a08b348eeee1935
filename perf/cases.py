"""Performance cases: what a user's program has the library do, through its public entry
points, on the workloads of this repository (cube 16^3, shield 64 x 64 x 96, lens 96^3 and
128^3, batched shields) and on ragged grids of the supported lengths.

Fields are float64 device arrays [component][z][y][x].  A context of FP32 passes computes the
values of curl, Phi, dh/dt and gradients in FP32 and hands them out in float64 arrays; a program
of that precision keeps such results as float32, and so do the FP32 cases here.

States are what a run holds between ramps: a current of at most about 0.85 jc in the solid (an
azimuthal part and a smooth random part) and its field h = Phi[j] + h_e, so the power law is
neither idle nor at the critical point, where dh/dt amplifies any rounding by some thousands.

The reference values of `exact` are plain 64-bit torch: library FFTs, the zero-padded
convolution, the fixed-point iteration, the Bogacki-Shampine pair, and torch's own gradients.
"""

from __future__ import annotations

import math
import random

import numpy as np
import torch

import paper_1803_01346_gb300 as S
import scfft_inputs as I

PREC = {"f64": S.PREC_F64, "f32": S.PREC_F32, "df64": S.PREC_DF64}
SIZES = (16, 32, 48, 64, 96, 128)
DEV = "cuda"


# ----------------------------------------------------------------------------
# the cases
# ----------------------------------------------------------------------------
def _case(op, prec, n, solid, **more):
    return {"op": op, "prec": prec, "nx": n[0], "ny": n[1], "nz": n[2], "solid": solid, **more}


def listed():
    return [
        # the current density of a snapshot of the smallest workload: the shortest call there is
        {"name": "curl_cube16_f64", **_case("curl", "f64", (16, 16, 16), "cube")},
        # the plain FP64 run of the cube: adaptive steps with two snapshots, host-driven, launch-bound
        {"name": "integrate_cube16_f64", **_case("integrate", "f64", (16, 16, 16), "cube", dt=2e-3, span=3e-2)},
        # one right-hand side of the shield in each arithmetic (a program with its own integrator)
        {"name": "rhs_shield_f64", **_case("rhs", "f64", (64, 64, 96), "shield")},
        {"name": "rhs_shield_f32", **_case("rhs", "f32", (64, 64, 96), "shield")},
        {"name": "rhs_shield_df64", **_case("rhs", "df64", (64, 64, 96), "shield")},
        # the Biot-Savart field alone (post-processing), FP64 at the adjoint workload's grid and
        # FP32 on a ragged one whose axes use three different transforms
        {"name": "phi_lens96_f64", **_case("phi", "f64", (96, 96, 96), "lens")},
        {"name": "phi_ragged_f32", **_case("phi", "f32", (48, 32, 128), "cube")},
        # the lens at full size: one right-hand side, and device-resident steps after a restart
        {"name": "rhs_lens128_f32", **_case("rhs", "f32", (128, 128, 128), "lens")},
        {"name": "advance_lens128_f32", **_case("advance", "f32", (128, 128, 128), "lens", dt=1e-7, steps=4)},
        # reverse mode: the gradient of the lens with its jc map, and the FP64 one on a copy
        {"name": "vjp_lens96_f32", **_case("vjp", "f32", (96, 96, 96), "lens", iters=5, jc=True)},
        {"name": "vjp_shield48_f64", **_case("vjp", "f64", (48, 48, 48), "shield", iters=5, jc=False)},
        # independent shields of uneven grids advanced together
        {"name": "batch_shields_f32", "op": "batch", "prec": "f32", "count": 12, "batch_seed": 1803, "dt": 2e-7,
         "steps": 3},
    ]


def draw(rng: random.Random):
    op = rng.choice(["curl", "phi", "phi", "rhs", "rhs", "rhs", "advance", "integrate", "vjp", "vjp", "batch"])
    prec = rng.choice(["f32", "f32", "f64", "df64"])
    solid = rng.choice(["cube", "shield", "lens"])
    # (a pass of FP64 transforms costs about 25 times the FP32 one, so its grids end earlier)
    most = {"f32": 128 ** 3, "df64": 96 ** 3, "f64": 96 * 96 * 64}[prec]
    if op == "batch":
        return {"op": "batch", "prec": "f32", "count": rng.randint(2, 10), "batch_seed": rng.randrange(1000),
                "dt": 10.0 ** rng.uniform(-7.5, -7.0), "steps": rng.randint(1, 3)}
    if op == "integrate":
        n = tuple(rng.choice((16, 32)) for _ in range(3))
        return _case(op, prec, n, "cube", dt=1e-3 * rng.uniform(1.0, 2.0), span=1e-2 * rng.uniform(1.0, 2.0))
    while True:
        n = tuple(rng.choice(SIZES) for _ in range(3))
        if n[0] * n[1] * n[2] <= most:
            break
    if op == "advance":
        return _case(op, "f32", n, solid, dt=10.0 ** rng.uniform(-7.5, -7.0), steps=rng.randint(1, 4))
    if op == "vjp":
        return _case(op, prec, n, solid, iters=rng.randint(2, 5), jc=rng.random() < 0.5)
    return _case(op, prec, n, solid, amp=rng.uniform(0.6, 0.85))


# ----------------------------------------------------------------------------
# workloads
# ----------------------------------------------------------------------------
def _grid(case):
    return (case["nx"], case["ny"], case["nz"])


def _config(case):
    """Box, solid and material of a case (the repository's own workloads, scaled to its grid)."""
    name = {"cube": "cube16", "shield": "shield64x64x96", "lens": "lens128"}[case["solid"]]
    c = I.config(name, scale=_grid(case))
    if case["solid"] == "cube":
        c.L = (1.6, 1.6, 1.6)  # (a margin of two nodes on every grid)
        c.mask = I.cube(c.n, c.L, 1.6)
    if case["solid"] == "shield":
        c.L = (1.6, 1.6, 2.4)
        c.mask = I.shield(c.n, c.L, 1.0, 0.6, 3.0, 0.4)
    if case["solid"] == "lens":
        c.mask = I.lens(c.n, c.L, 1.0, 1.0, 0.15, 0.05)
    return c


def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed))
    return g


class Box:
    """Grid, symbols and kernel spectrum of the method in plain 64-bit torch."""

    def __init__(self, n, L):
        self.n, self.L = n, L
        nx, ny, nz = n
        self.d = tuple(2.0 * a / k for a, k in zip(L, n))
        self.sigma = 0.5 * math.sqrt(sum(v * v for v in self.d))
        ks, ds = [], []
        for k, a in zip(n, L):
            m = torch.fft.fftfreq(k, d=1.0 / k, dtype=torch.float64, device=DEV) * (math.pi / a)
            dv = m.clone()
            dv[k // 2] = 0.0
            ks.append(m)
            ds.append(dv)
        kx, dx = ks[0][: nx // 2 + 1], ds[0][: nx // 2 + 1]
        k2 = kx[None, None, :] ** 2 + ks[1][None, :, None] ** 2 + ks[2][:, None, None] ** 2
        self.S = torch.exp(-0.5 * self.sigma ** 2 * k2)
        self.D = (dx[None, None, :], ds[1][None, :, None], ds[2][:, None, None])
        self._K = None

    def smooth(self, f, cells):
        s = cells * max(self.d)
        return torch.fft.irfftn(torch.fft.rfftn(f, dim=(1, 2, 3)) * self.S ** (2 * s * s / self.sigma ** 2),
                                s=f.shape[1:], dim=(1, 2, 3))

    def curl(self, f):
        F = torch.fft.rfftn(f, dim=(1, 2, 3))
        x, y, z = self.D
        G = torch.stack([(y * F[2] - z * F[1]) * self.S, (z * F[0] - x * F[2]) * self.S,
                         (x * F[1] - y * F[0]) * self.S])
        return torch.fft.irfftn(1j * G, s=f.shape[1:], dim=(1, 2, 3))

    def kernel(self):
        if self._K is None:
            nx, ny, nz = self.n
            off = [torch.fft.fftfreq(2 * k, d=1.0 / (2 * k), dtype=torch.float64, device=DEV) * dv
                   for k, dv in zip(self.n, self.d)]
            X, Y, Z = off[0][None, None, :], off[1][None, :, None], off[2][:, None, None]
            r = torch.sqrt(X * X + Y * Y + Z * Z)
            r[0, 0, 0] = 1.0
            u = r / (math.sqrt(2.0) * self.sigma)
            g = (2.0 / math.sqrt(math.pi) * u * torch.exp(-u * u) - torch.erf(u)) / (4.0 * math.pi * r ** 3)
            g[0, 0, 0] = 0.0
            g[:, :, nx] = 0.0
            g[:, ny, :] = 0.0
            g[nz, :, :] = 0.0
            dV = self.d[0] * self.d[1] * self.d[2]
            self._K = [torch.fft.rfftn(dV * g * c) for c in (X, Y, Z)]
        return self._K

    def phi(self, j):
        nx, ny, nz = self.n
        J = torch.fft.rfftn(j, s=(2 * nz, 2 * ny, 2 * nx), dim=(1, 2, 3))
        K = self.kernel()
        out = []
        for a in range(3):
            b, c = (a + 1) % 3, (a + 2) % 3
            P = torch.fft.irfftn(K[b] * J[c] - K[c] * J[b], s=(2 * nz, 2 * ny, 2 * nx))
            out.append(P[:nz, :ny, :nx])
        return torch.stack(out)


def _fields(case, cfg, seed, amp=0.85):
    """(h, j, g): field, current and warm start of a state made from the seed.  The current falls
    off within about a cell of the solid's surface, as the stray current outside makes it do in a
    run, and the warm start is dh/dt of a state with a little less current: the state before."""
    gen = _gen(seed)
    m = Method(cfg, None, 0.0, 10)
    box = m.box
    nx, ny, nz = cfg.n
    x, y, _ = (torch.from_numpy(v).to(DEV) for v in I.node_axes(cfg.n, cfg.L))
    j = box.smooth(torch.randn((3, nz, ny, nx), generator=gen, dtype=torch.float64, device=DEV), 1.5)
    j = 0.3 * j / j.abs().max()
    j[0] -= y[None, :, None]
    j[1] += x[None, None, :]
    inside = m.mask.to(torch.float64)
    j = j * (inside * (2.0 * box.smooth(inside[None], 0.7)[0] - 1.0).clamp(min=0.0))
    j = j * (amp / torch.sqrt((j * j).sum(0)).max())
    he = torch.tensor([0.02, -0.03, 0.1], dtype=torch.float64, device=DEV)[:, None, None, None]
    h = box.phi(j)
    rate = torch.tensor(_rate(cfg), dtype=torch.float64, device=DEV)
    g = m.rhs(he + 0.995 * h, rate[:, None, None, None].expand(h.shape), rate)
    return (h + he).contiguous(), j.contiguous(), g.contiguous()


def _rate(cfg):
    """dh_e/dt on the first ramp."""
    return [float(a) / cfg.knots_t[1] for a in cfg.knots_he[1]]


# device-resident FP32 steps start small after a restart and grow by the controller's limit of five
# a step; this tolerance leaves the limit in charge, not FP32 rounding of the error estimate
ATOL = 1e-3
T0 = 0.05  # every state stands at this time, on the first ramp


def _context(cfg, prec, stream=None, delta_it=2e-5, max_iter=100, rtol=None, atol=None):
    ctx = S.Context(cfg.n, cfg.L, n_power=cfg.n_power, rho_out=cfg.rho_out, precision=PREC[prec], delta_it=delta_it,
                    max_iter=max_iter, rtol=rtol or cfg.rtol, atol=atol or cfg.atol, stream=stream)
    ctx.set_geometry(cfg.mask)
    ctx.set_field_path(cfg.knots_t, cfg.knots_he)
    ctx.precompute_kernel()
    return ctx


def _jc(cfg, seed):
    nx, ny, nz = cfg.n
    u = torch.rand((nz, ny, nx), generator=_gen(seed + 77), dtype=torch.float64, device=DEV)
    return 0.95 + 0.1 * u


# one batch of contexts is kept for the whole program, as a program that advances a batch keeps it:
# its states are inputs copied into the batch's own buffers
_batch: dict = {}


def _batch_of(case):
    key = tuple(sorted((k, v) for k, v in case.items() if k != "name"))
    if _batch.get("key") != key:
        _batch.clear()
        cfgs = I.batch_configs(case["count"], seed=case["batch_seed"])
        # (on one stream: inputs are copied into the batch's buffers in the order of the program)
        _batch.update(key=key, cfgs=cfgs, ctxs=[_context(c, case["prec"], atol=ATOL) for c in cfgs],
                      h=[torch.empty(3 * int(np.prod(c.n)), dtype=torch.float64, device=DEV) for c in cfgs],
                      w=[torch.empty(3 * int(np.prod(c.n)), dtype=torch.float64, device=DEV) for c in cfgs])
        for c in _batch["ctxs"]:
            c.autotune()
    return dict(_batch)


def prepare(case, seed):
    if case["op"] == "batch":
        b = _batch_of(case)
        ins = [_fields(case, c, seed * 101 + i, 0.7) for i, c in enumerate(b["cfgs"])]
        return {"case": case, **b, "h0": [v[0].reshape(-1) for v in ins], "w0": [v[2].reshape(-1) for v in ins]}
    cfg = _config(case)
    h, j, g = _fields(case, cfg, seed, case.get("amp", 0.85))
    fixed = {"delta_it": 0.0, "max_iter": case["iters"]} if case["op"] == "vjp" else {}
    if case["op"] == "integrate":
        fixed = {"rtol": 1e-6}
    if case["op"] == "advance":
        fixed = {"atol": ATOL}
    ctx = _context(cfg, case["prec"], **fixed)
    n3 = h.numel()

    def empty(k=n3):
        return torch.empty(k, dtype=torch.float64, device=DEV)

    s = {"case": case, "ctx": ctx, "h0": h.reshape(-1), "g0": g.reshape(-1), "h": empty(), "w": empty(), "out": empty()}
    if case["op"] == "advance":
        ctx.autotune()
    if case["op"] == "phi":
        s["h0"] = (j + 0.05 * torch.randn(j.shape, generator=_gen(seed + 5), dtype=torch.float64, device=DEV)).reshape(-1)
    if case["op"] == "integrate":
        s["snaps"] = empty(2 * n3)
    if case["op"] == "vjp":
        s["lam"] = torch.randn(n3, generator=_gen(seed + 9), dtype=torch.float64, device=DEV)
        s["mu_g"], s["mu_jc"] = empty(), empty(n3 // 3) if case["jc"] else None
        if case["jc"]:
            ctx.set_jc_map(_jc(cfg, seed).reshape(-1).contiguous())
    return s


# ----------------------------------------------------------------------------
# one pass
# ----------------------------------------------------------------------------
def _kept(case, x):
    """A result as a program of the case's precision keeps it."""
    return x.float() if case["prec"] == "f32" else x


def run(s):
    case = s["case"]
    op = case["op"]
    if op == "batch":
        for a, b in zip(s["h"] + s["w"], s["h0"] + s["w0"]):
            a.copy_(b)
        nb = len(s["ctxs"])
        t, dt, stop = [T0] * nb, [case["dt"]] * nb, [1.0] * nb
        for _ in range(case["steps"]):
            t, dt, st = S.batch_step(s["ctxs"], t, dt, stop, s["h"], s["w"])
        return {"h": [_kept(case, x) for x in s["h"]], "w": [_kept(case, x) for x in s["w"]], "t": np.array(t),
                "dt": np.array(dt), "status": np.array(st)}
    ctx = s["ctx"]
    if op == "curl":
        ctx.curl(s["h0"], s["out"])
        return _kept(case, s["out"])
    if op == "phi":
        ctx.phi(s["h0"], s["out"])
        return _kept(case, s["out"])
    if op == "rhs":
        s["w"].copy_(s["g0"])  # the call replaces the warm start by its result
        ctx.rhs(T0, s["h0"], s["w"], s["out"])
        return _kept(case, s["out"])
    if op == "advance":
        s["h"].copy_(s["h0"])
        s["w"].copy_(s["g0"])
        t, dt, n = ctx.advance(T0, case["dt"], 1.0, case["steps"], s["h"], s["w"])
        return {"h": _kept(case, s["h"]), "w": _kept(case, s["w"]), "t": np.array([t, dt]), "n": n}
    if op == "integrate":
        s["h"].copy_(s["h0"])
        s["w"].copy_(s["g0"])
        t1 = T0 + case["span"]
        st = ctx.integrate(T0, t1, case["dt"], s["h"], tsnap=[T0 + 0.5 * case["span"], t1], snaps=s["snaps"],
                           warm=s["w"])
        return {"h": _kept(case, s["h"]), "snaps": _kept(case, s["snaps"]), "w": _kept(case, s["w"]), "t": st["t"]}
    assert op == "vjp"
    mu_a = ctx.rhs_vjp(s["h0"], s["lam"], s["out"], s["mu_g"], s["mu_jc"])
    return {"h": _kept(case, s["out"]), "g": _kept(case, s["mu_g"]), "a": mu_a,
            "jc": _kept(case, s["mu_jc"]) if case["jc"] else []}


# ----------------------------------------------------------------------------
# the work of a pass
# ----------------------------------------------------------------------------
def _fft(length):
    return 5.0 * length * math.log2(length)


def _curl_flops(n):
    """Three real transforms forward, three back, on the grid."""
    nx, ny, nz = n
    h = nx // 2 + 1
    return 6 * (0.5 * ny * nz * _fft(nx) + h * nz * _fft(ny) + h * ny * _fft(nz))


def _phi_flops(n):
    """The same on the doubled grid, over the pencils that hold anything or are kept."""
    nx, ny, nz = n
    h = nx + 1
    return 6 * (0.5 * ny * nz * _fft(2 * nx) + h * nz * _fft(2 * ny) + h * 2 * ny * _fft(2 * nz))


ITERS = 5  # iterations of a right-hand side that stops by its tolerance, about


def work(case):
    op = case["op"]
    if op == "batch":
        b = f = 0.0
        for c in I.batch_configs(case["count"], seed=case["batch_seed"]):
            N = float(np.prod(c.n))
            b += 97 * N
            f += (1 + 3 * case["steps"]) * (2 * _curl_flops(c.n) + ITERS * (_curl_flops(c.n) + _phi_flops(c.n)))
        return {"bytes": b, "flops": f}
    n = _grid(case)
    N = float(n[0] * n[1] * n[2])
    c, p = _curl_flops(n), _phi_flops(n)
    rhs = 2 * c + ITERS * (c + p)
    if op == "curl":
        return {"bytes": 48 * N, "flops": c}
    if op == "phi":
        return {"bytes": 48 * N, "flops": p}
    if op == "rhs":
        return {"bytes": 97 * N, "flops": rhs}
    if op == "advance":
        return {"bytes": 97 * N, "flops": (1 + 3 * case["steps"]) * rhs}
    if op == "integrate":
        return {"bytes": 145 * N, "flops": (1 + 3 * case["span"] / case["dt"]) * rhs}
    return {"bytes": (24 * 4 + 1 + (16 if case["jc"] else 0)) * N, "flops": case["iters"] * (c + p) + 3 * c}


# ----------------------------------------------------------------------------
# reference values
# ----------------------------------------------------------------------------
class Method:
    def __init__(self, cfg, jc=None, delta_it=2e-5, max_iter=100):
        self.box, self.cfg, self.jc, self.delta_it, self.max_iter = Box(cfg.n, cfg.L), cfg, jc, delta_it, max_iter
        self.mask = torch.from_numpy(np.ascontiguousarray(cfg.mask)).to(DEV)
        self.out = int((~self.mask).sum())

    def rate(self, t):
        r = [0.0] * 3
        kt, kh = self.cfg.knots_t, self.cfg.knots_he
        for a in range(len(kt) - 1):
            if kt[a] <= t < kt[a + 1]:
                r = [(kh[a + 1][q] - kh[a][q]) / (kt[a + 1] - kt[a]) for q in range(3)]
        return r

    def rhs(self, h, g, rate):
        """dh/dt; rate: a tensor of three values."""
        cfg, box, m = self.cfg, self.box, self.mask
        j = box.curl(h)
        jn = torch.sqrt((j * j).sum(0))
        jc = 1.0 if self.jc is None else self.jc
        rho = torch.where(m, (jn / jc) ** (cfg.n_power - 1.0) / jc, torch.full_like(jn, cfg.rho_out))
        d = torch.where(m, -box.curl(rho * j), g)
        tol = self.delta_it * max(float(rate.detach().norm()), 1.0)
        for _ in range(self.max_iter):
            new = torch.where(m, d, rate[:, None, None, None] + box.phi(box.curl(d) * m))
            if self.delta_it > 0:
                res = float((torch.sqrt(((new - d) ** 2).sum(0)) * ~m).sum()) / self.out
                d = new
                if res < tol:
                    break
            else:
                d = new
        return d

    def at(self, t, h, g):
        return self.rhs(h, g, torch.tensor(self.rate(t), dtype=torch.float64, device=DEV))

    def steps(self, h, g, dt, t1, nsteps, stops, rtol, atol):
        """Accepted Bogacki-Shampine steps from T0: (h, last dh/dt, t, dt, steps, states at the stops)."""
        t, seen = T0, []
        k1 = self.at(t, h, g)
        last, n = k1, 0
        ends = [v for v in list(stops) + [t1] if v > T0]
        while n < nsteps and t < t1:
            nxt = min([v for v in ends if v > t])
            while True:
                hs = min(dt, nxt - t)
                hits = hs == nxt - t
                k2 = self.at(t + 0.5 * hs, h + hs * 0.5 * k1, last)
                k3 = self.at(t + 0.75 * hs, h + hs * 0.75 * k2, k2)
                new = h + hs * (2 / 9 * k1 + 1 / 3 * k2 + 4 / 9 * k3)
                k4 = self.at(nxt if hits else t + hs, new, k3)
                last = k4
                e = hs * ((2 / 9 - 7 / 24) * k1 + (1 / 3 - 1 / 4) * k2 + (4 / 9 - 1 / 3) * k3 - k4 / 8)
                w = torch.clamp(rtol * torch.maximum(h.abs(), new.abs()), min=atol)
                err = float((e.abs() / w).max())
                if err <= 1.0:
                    break
                dt = hs * max(0.2, 0.9 * err ** (-1 / 3))
            h, k1, t, n = new, k4, (nxt if hits else t + hs), n + 1
            dt = hs * (5.0 if err == 0 else min(5.0, max(0.2, 0.9 * err ** (-1 / 3))))
            if hits and nxt in stops:
                seen.append(h)
        return h, last, t, dt, n, seen


def exact(case, seed):
    op = case["op"]
    if op == "batch":
        hs, ws, ts, dts = [], [], [], []
        for i, c in enumerate(I.batch_configs(case["count"], seed=case["batch_seed"])):
            h, _, g = _fields(case, c, seed * 101 + i, 0.7)
            h, w, t, dt, _, _ = Method(c).steps(h, g, case["dt"], 1.0, case["steps"], (), c.rtol, ATOL)
            hs.append(h.reshape(-1))
            ws.append(w.reshape(-1))
            ts.append(t)
            dts.append(dt)
        return {"h": hs, "w": ws, "t": np.array(ts), "dt": np.array(dts),
                "status": np.zeros(case["count"], dtype=np.int64)}
    cfg = _config(case)
    h, j, g = _fields(case, cfg, seed, case.get("amp", 0.85))
    if op == "curl":
        return Box(cfg.n, cfg.L).curl(h).reshape(-1)
    if op == "phi":
        j = j + 0.05 * torch.randn(j.shape, generator=_gen(seed + 5), dtype=torch.float64, device=DEV)
        return Box(cfg.n, cfg.L).phi(j).reshape(-1)
    if op == "rhs":
        return Method(cfg).at(T0, h, g).reshape(-1)
    if op == "advance":
        h, w, t, dt, n, _ = Method(cfg).steps(h, g, case["dt"], 1.0, case["steps"], (), cfg.rtol, ATOL)
        return {"h": h.reshape(-1), "w": w.reshape(-1), "t": np.array([t, dt]), "n": n}
    if op == "integrate":
        t1 = T0 + case["span"]
        h, w, t, _, _, seen = Method(cfg).steps(h, g, case["dt"], t1, 10 ** 6, (T0 + 0.5 * case["span"], t1), 1e-6, cfg.atol)
        return {"h": h.reshape(-1), "snaps": torch.cat([v.reshape(-1) for v in seen]), "w": w.reshape(-1), "t": t}
    jc = _jc(cfg, seed) if case["jc"] else None
    m = Method(cfg, jc, 0.0, case["iters"])
    rate = torch.tensor(m.rate(T0), dtype=torch.float64, device=DEV)
    ins = [h.requires_grad_(), g.requires_grad_(), rate.requires_grad_()] + ([jc.requires_grad_()] if case["jc"] else [])
    lam = torch.randn(h.numel(), generator=_gen(seed + 9), dtype=torch.float64, device=DEV).reshape(h.shape)
    gr = torch.autograd.grad((m.rhs(h, g, rate) * lam).sum(), ins)
    return {"h": gr[0].reshape(-1), "g": gr[1].reshape(-1), "a": [float(v) for v in gr[2]],
            "jc": gr[3].reshape(-1) if case["jc"] else []}

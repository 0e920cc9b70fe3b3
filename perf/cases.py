"""The work that users of libmrcm have it do, as measured cases.

A case is a problem (grid, permeability field, boundary data), the method's parameters and the call
that a program makes on it (``kind``):

  operator  w = A v on a factored handle (mrcm_apply_operator)
  precond   z = T r on a factored handle (mrcm_apply_precond), as a program's own Krylov loop calls it
  setup     a new permeability field for a handle, its set-up (mrcm_factor_local) and one z = T r
  solve     set-up and GMRES from p0 = 0 (mrcm_factor_local, mrcm_gmres_solve)
  source    GMRES with another right-hand side on a handle that stays factored
  host      K from pinned host memory, p back to it (mrcm_solve_host)
  serve     a burst of requests through the request server (Server.submit, Server.poll)

All inputs are made from the seed on the GPU.  Solves with FP32 local factors run to 1e-11: a pressure
converged that far is the problem's own, whatever the rounding of the local solves that led to it.
"""

import ctypes as C
import math
import time

import numpy as np
import torch

from paper_2606_08883_gb300 import mrcm
from paper_2606_08883_gb300 import workloads as W

F8 = torch.float64
PAGE = 1 << 21
DEFAULTS = dict(ny=0, sub=32, l=2, sweeps=1, prec=W.PREC_FP64, refine=0, degree=0, mult=0, tensor=0, field="lognormal",
                var=4.0, corr=0.05, tol=1e-8, fluxes=0, requests=0, inflight=8)


def listed():
    return [
        # the smallest call: one stencil on the 64^2 grid of the quarter-five-spot problem
        dict(name="operator-64", kind="operator", nx=64, sub=16, field="spot", var=2.0, corr=0.1),
        # the operator at the benchmark's size, where it streams 134 MB
        dict(name="operator-2048", kind="operator", nx=2048, prec=W.PREC_FP32),
        # T on 16 small boxes: launches and dependent steps
        dict(name="precond-spot-64", kind="precond", nx=64, sub=16, field="spot", var=2.0, corr=0.1),
        # T in FP64 as in the 512^2 channel workload: 40-wide boxes, two sweeps
        dict(name="precond-channels-512", kind="precond", nx=512, l=4, sweeps=2, field="channels"),
        # T in FP64 on a large grid: 1,024 boxes 36 wide
        dict(name="precond-lognormal-1024", kind="precond", nx=1024),
        # the variants together: a grid that the subdomains do not divide, tensor K, piecewise-linear
        # interface spaces, multiplicative sweeps; set-up and one application
        dict(name="setup-variants-461x333", kind="setup", nx=461, ny=333, sub=24, l=3, degree=1, mult=1, tensor=1,
             field="random", var=3.0),
        # the smallest whole solve, with the fluxes that a transport code takes
        dict(name="solve-spot-64", kind="solve", nx=64, sub=16, field="spot", var=2.0, corr=0.1, fluxes=1),
        # the FP64 workload: 512^2 channels of contrast 1e6
        dict(name="solve-channels-512", kind="solve", nx=512, l=4, sweeps=2, field="channels"),
        # the benchmark's default workload, FP32 local solves inside FP64 GMRES
        dict(name="solve-mixed-2048", kind="solve", nx=2048, prec=W.PREC_FP32, refine=2, tol=1e-11),
        # a time step or another well pattern on the same field: GMRES alone
        dict(name="source-mixed-1024", kind="source", nx=1024, prec=W.PREC_FP32, refine=2, corr=0.1, tol=1e-11),
        # one member of an ensemble whose fields and answers live on the host
        dict(name="host-mixed-512", kind="host", nx=512, prec=W.PREC_FP32, refine=2, corr=0.1, tol=1e-11),
        # a burst at the server: grids of 128^2, 256^2 and 512^2 in turn
        dict(name="serve-9", kind="serve", nx=512, prec=W.PREC_FP32, refine=2, corr=0.1, tol=1e-11, requests=9),
    ]


def _side(rng, lo, hi, sub, l):
    """Cells of one axis, spread over the logarithm; the last subdomain stays wider than the oversampling."""
    n = int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))
    rest = n % sub
    return n if rest == 0 or rest > max(l, 1) else n - rest


def draw(rng):
    kind = rng.choice(["operator", "precond", "precond", "setup", "solve", "solve", "source", "host"])
    mixed = rng.random() < 0.5
    sub, l = rng.choice([16, 20, 24, 32]), rng.choice([2, 3, 4])
    case = dict(kind=kind, sub=sub, l=l, sweeps=rng.choice([1, 2]), field=rng.choice(["lognormal", "channels", "random"]))
    if case["field"] == "channels":   # contrast 1e6: FP64 and the wider overlap, as in the 512^2 workload
        case.update(sub=32, l=4, sweeps=2)
        mixed = False
    elif case["field"] == "random":
        case.update(var=round(rng.uniform(1.0, 3.0), 3))
    else:
        case.update(var=round(rng.uniform(1.0, 4.0), 3), corr=round(rng.uniform(0.05, 0.15), 3))
    hi = {"operator": 2048, "precond": 1024}.get(kind, 640)
    if kind in ("precond", "setup"):  # the multiscale solution itself, in the precision of its storage
        mixed = False
        case.update(degree=rng.choice([0, 0, 1]), mult=rng.choice([0, 0, 1]), tensor=rng.choice([0, 1]))
        hi = 640 if case["degree"] else hi
    case["nx"] = _side(rng, 64, hi, case["sub"], case["l"])
    case["ny"] = _side(rng, max(64, case["nx"] // 3), min(hi, 3 * case["nx"]), case["sub"], case["l"])
    if mixed:
        case.update(prec=W.PREC_FP32, refine=rng.choice([1, 2]), tol=1e-11)
    return case


# ------------------------------------------------------------------------------------------ inputs

def _full(case):
    c = dict(DEFAULTS, **case)
    c["ny"] = c["ny"] or c["nx"]
    return c


def _gaussian(ny, nx, h, corr, var, gen):
    """Stationary Gaussian field with exponential covariance by circulant embedding, negative
    eigenvalues clipped (Dietrich and Newsam, 1997)."""
    my, mx = 2 * ny, 2 * nx
    dy = torch.arange(my, device="cuda", dtype=F8)
    dx = torch.arange(mx, device="cuda", dtype=F8)
    dy, dx = torch.minimum(dy, my - dy) * (h / corr), torch.minimum(dx, mx - dx) * (h / corr)
    lam = torch.fft.fft2(var * torch.exp(-torch.hypot(dy[:, None], dx[None, :]))).real.clamp_min(0.0)
    xi = torch.randn(2, my, mx, generator=gen, device="cuda", dtype=F8)
    return torch.fft.fft2(torch.sqrt(lam / lam.numel()) * torch.complex(xi[0], xi[1])).real[:ny, :nx].contiguous()


def _channels(ny, nx, h, gen):
    """Sinuous channels of permeability 1e6 along x until they fill 30 % of the cells."""
    x, y = (torch.arange(nx, device="cuda", dtype=F8) + 0.5) * h, (torch.arange(ny, device="cuda", dtype=F8) + 0.5) * h
    mask = torch.zeros(ny, nx, dtype=torch.bool, device="cuda")
    while float(mask.double().mean()) < 0.3:
        u = torch.rand(5, generator=gen, device="cuda", dtype=F8)
        at = u[0] * ny * h + (0.02 + 0.08 * u[1]) * torch.sin(2 * math.pi * (x / (0.2 + 0.4 * u[2]) + u[3]))
        mask |= (y[:, None] - at[None, :]).abs() < 0.5 * (0.01 + 0.02 * u[4])
    return torch.where(mask, 1e6, 1.0).to(F8)


def _problem(c, seed):
    """Permeability components [1 or 2, ny, nx], source, boundary pressures on the x sides, and cell size."""
    nx, ny = c["nx"], c["ny"]
    h = 1.0 / max(nx, ny)
    gen = torch.Generator(device="cuda").manual_seed(int(seed))
    comp = []
    for _ in range(2 if c["tensor"] else 1):
        if c["field"] == "channels":
            comp.append(_channels(ny, nx, h, gen))
        elif c["field"] == "random":   # independent cells, contrast 10^var
            comp.append(10.0 ** (c["var"] * torch.rand(ny, nx, generator=gen, device="cuda", dtype=F8)))
        else:
            comp.append(torch.exp(_gaussian(ny, nx, h, c["corr"], c["var"], gen)))
    f, left = None, torch.ones(ny, device="cuda", dtype=F8)
    if c["field"] == "spot":           # quarter five-spot: wells in opposite corners, p = 0 on both sides
        f, left = torch.zeros(ny, nx, device="cuda", dtype=F8), 0.0 * left
        f[0, 0], f[-1, -1] = 1.0, -1.0
    elif c["kind"] == "source":        # distributed sources besides the pressure drop
        f = torch.randn(ny, nx, generator=gen, device="cuda", dtype=F8) * h * h
    vec = torch.randn(ny * nx, generator=gen, device="cuda", dtype=F8)
    return torch.stack(comp), f, left, vec / vec.norm(), h


def _params(c):
    return W.Params(sub=(c["sub"], c["sub"], 1), oversample=c["l"], smooth_steps=c["sweeps"], alpha=10.0, tol=c["tol"],
                    restart=30, max_iter=300, local_prec=c["prec"], smooth_kind=c["mult"], iface_degree=c["degree"],
                    refine_setup=c["refine"])


# --------------------------------------------------------------------------------------- the calls

class Handle:
    """A libmrcm handle on this program's own workspace, which it takes in whole pages, one to spare."""

    def __init__(self, c, seed):
        self.c = c
        K, f, left, self.v, h = _problem(c, seed)
        self.K, self.f, self.bc = K, f, [left, torch.zeros_like(left)]
        dirichlet_x = [W.DIRICHLET, W.DIRICHLET] + 4 * [W.NEUMANN]
        grid = W.Problem(2, (c["nx"], c["ny"], 1), (h, h, 1.0), None, dirichlet_x)
        self.p = mrcm.make_problem(grid, K[0].data_ptr(), [b.data_ptr() for b in self.bc] + 4 * [0],
                                   0 if f is None else f.data_ptr(), K[1].data_ptr() if len(K) > 1 else 0)
        self.q = mrcm.make_params(_params(c))
        need = mrcm.footprint(grid, _params(c))
        self.ws = torch.empty((need // PAGE + 2) * PAGE, dtype=torch.uint8, device="cuda")
        self.h, self.res = C.c_void_p(), mrcm.mrcm_result()
        self.ok(mrcm.mrcm_setup(C.byref(self.p), C.byref(self.q), self.ws.data_ptr(), self.ws.numel(), self.stream(),
                                C.byref(self.h)))
        n = c["nx"] * c["ny"]
        self.out = torch.zeros(n, device="cuda", dtype=F8)
        if c["kind"] == "host":
            self.host_K = K[0].cpu().pin_memory()
            self.host_p = torch.empty(n, dtype=F8, pin_memory=True)
        if c["fluxes"]:
            self.u = [torch.empty((c["nx"] + 1) * c["ny"], device="cuda", dtype=F8),
                      torch.empty(c["nx"] * (c["ny"] + 1), device="cuda", dtype=F8)]
        if c["kind"] in ("operator", "precond", "source"):
            self.factor()
        if c["kind"] == "source":
            self.b = torch.empty(n, device="cuda", dtype=F8)
            self.ok(mrcm.mrcm_rhs(self.h, self.b.data_ptr(), self.stream()))

    @staticmethod
    def stream():
        return torch.cuda.current_stream().cuda_stream

    def ok(self, rc):
        if rc != mrcm.MRCM_OK:
            raise mrcm.MRCMError(rc, (mrcm.mrcm_last_error(self.h or None) or b"").decode())

    def factor(self):
        self.ok(mrcm.mrcm_factor_local(self.h, self.stream()))

    def run(self):
        c, out = self.c, self.out
        if c["kind"] == "operator":
            self.ok(mrcm.mrcm_apply_operator(self.h, self.v.data_ptr(), out.data_ptr(), self.stream()))
            return out
        if c["kind"] == "host":
            self.ok(mrcm.mrcm_solve_host(self.h, self.host_K.data_ptr(), self.host_p.data_ptr(), C.byref(self.res),
                                         self.stream()))
            return self.host_p
        if c["kind"] == "setup":
            self.ok(mrcm.mrcm_update_problem(self.h, C.byref(self.p), self.stream()))
        if c["kind"] in ("setup", "solve"):
            self.factor()
        if c["kind"] in ("setup", "precond"):
            self.ok(mrcm.mrcm_apply_precond(self.h, self.v.data_ptr(), out.data_ptr(), self.stream()))
            return out
        out.zero_()
        b = self.b.data_ptr() if c["kind"] == "source" else None
        ux, uy = [u.data_ptr() for u in self.u] if c["fluxes"] else (None, None)
        self.ok(mrcm.mrcm_gmres_solve(self.h, b, out.data_ptr(), ux, uy, None, C.byref(self.res), self.stream()))
        return [out] + self.u if c["fluxes"] else out

    def __del__(self):
        if getattr(self, "h", None):
            mrcm.mrcm_destroy(self.h)
            self.h = None


def _requests(c):
    """The requests of a burst: the case's grid, a half and a quarter of it in turn."""
    for i in range(c["requests"]):
        n = c["nx"] >> (2 - i % 3)
        yield dict(c, kind="solve", nx=n, ny=n, var=1.0 + (4.0 * i) / c["requests"])


class Burst:
    def __init__(self, c, seed):
        self.items = []
        room = 0
        for i, r in enumerate(_requests(c)):
            K, _, left, _, h = _problem(r, 1000 * seed + i)
            side = [v.cpu().numpy()[None] for v in (left, torch.zeros_like(left))]
            prob = W.Problem(2, (r["nx"], r["ny"], 1), (h, h, 1.0), K.cpu().numpy(),
                             [W.DIRICHLET, W.DIRICHLET] + 4 * [W.NEUMANN], side + 4 * [None])
            self.items.append((prob, _params(r)))
            room += mrcm.footprint(prob, _params(r)) + (64 << 20)
        self.server = mrcm.Server(room, max_inflight=c["inflight"])

    def run(self):
        waiting = {self.server.submit(prob, q): i for i, (prob, q) in enumerate(self.items)}
        out = [None] * len(self.items)
        while waiting:
            for t in list(waiting):
                got = self.server.poll(t)
                if got is not None:
                    rc, out[waiting.pop(t)], info = got
                    if rc != mrcm.MRCM_OK:
                        raise mrcm.MRCMError(rc, info.get("error", ""))
            time.sleep(2e-5)
        return out

    def __del__(self):
        if getattr(self, "server", None):
            self.server.close()


def prepare(case, seed):
    c = _full(case)
    return (Burst if c["kind"] == "serve" else Handle)(c, seed)


def run(state):
    return state.run()


# ------------------------------------------------------------------------------------------- work

def work(case):
    """Every array of the path read or written once, and the arithmetic of one line inverse per box
    line (w^3 flops), 2 w^2 flops per line product and about 12 flops per stencil; a solve to a
    relative residual tol is counted as 2 - log10(tol) steps."""
    c = _full(case)
    if c["kind"] == "serve":
        w = [work(dict(r, name="")) for r in _requests(c)]
        return {k: sum(x[k] for x in w) for k in ("bytes", "flops")}
    n, sub, l = c["nx"] * c["ny"], c["sub"], c["l"]
    S = -(-c["nx"] // sub) * -(-c["ny"] // sub)
    wide, elt, nq = sub + 2 * l, 4 if c["prec"] == W.PREC_FP32 else 8, 1 + c["degree"]
    box = elt * S * wide * wide * (wide + 1) // 2
    stencil = {"bytes": 8 * 4 * n, "flops": 12 * n}
    once = {"bytes": (1 + c["sweeps"]) * box + 8 * n * (3 + 4 * nq) + c["sweeps"] * 8 * 3 * n,
            "flops": S * (1 + c["sweeps"]) * 4 * wide ** 3 + n * (8 * nq + 12 * c["sweeps"])}
    setup = {"bytes": 2 * box + elt * S * sub * sub * (sub + 1) // 2 + 8 * n * (5 + 4 * nq),
             "flops": S * (2 * wide ** 4 + sub ** 4 + 16 * nq * (wide ** 3 + sub ** 3))}
    steps = 2 - math.log10(c["tol"])
    krylov = {"bytes": steps * (stencil["bytes"] + once["bytes"]) + 8 * n * steps * (steps + 2),
              "flops": steps * (stencil["flops"] + once["flops"]) + 3 * n * steps * (steps + 2)}
    parts = {"operator": [stencil], "precond": [once], "setup": [setup, once], "source": [krylov]}
    parts = parts.get(c["kind"], [setup, krylov])
    return {k: float(sum(p[k] for p in parts)) for k in ("bytes", "flops")}


# --------------------------------------------------------------- the same results in plain 64 bits

def _trans(c, K, h):
    """Two-point transmissibilities (ny, nx + 1) and (ny + 1, nx); p given on the x sides, no flow on the y sides."""
    Kx, Ky = K[0], K[-1]
    Tx = torch.zeros(c["ny"], c["nx"] + 1, device=K.device, dtype=F8)
    Ty = torch.zeros(c["ny"] + 1, c["nx"], device=K.device, dtype=F8)
    Tx[:, 1:-1] = 2 * Kx[:, :-1] * Kx[:, 1:] / (Kx[:, :-1] + Kx[:, 1:])
    Ty[1:-1] = 2 * Ky[:-1] * Ky[1:] / (Ky[:-1] + Ky[1:])
    Tx[:, 0], Tx[:, -1] = 2 * Kx[:, 0], 2 * Kx[:, -1]      # cells are square and of unit thickness
    return Tx, Ty


def _apply(Tx, Ty, v):
    g = torch.nn.functional.pad(v, (1, 1, 1, 1))
    m = g[1:-1, 1:-1]
    return Tx[:, 1:] * (m - g[1:-1, 2:]) + Tx[:, :-1] * (m - g[1:-1, :-2]) + Ty[1:] * (m - g[2:, 1:-1]) + \
        Ty[:-1] * (m - g[:-2, 1:-1])


class Lines:
    """Direct solver of B five-point systems (B, h, w): block elimination line by line with dense inverses."""

    def __init__(self, d, east, north):
        self.e, self.inv = north, []
        off = torch.diag_embed(east, 1) + torch.diag_embed(east, -1)
        for j in range(d.shape[1]):
            D = torch.diag_embed(d[:, j]) - off[:, j]
            if j:
                e = self.e[:, j - 1]
                D -= e[:, :, None] * self.inv[-1] * e[:, None, :]
            self.inv.append(torch.linalg.inv(D))

    def solve(self, b):
        y, x = [], [None] * len(self.inv)
        for j, S in enumerate(self.inv):
            t = b[:, j]
            if j:
                t = t + self.e[:, j - 1, :, None] * y[-1]
            y.append(S @ t)
        for j in reversed(range(len(x))):
            x[j] = y[j] if j + 1 == len(x) else y[j] + self.inv[j] @ (self.e[:, j, :, None] * x[j + 1])
        return torch.stack(x, 1)


class Multiscale:
    """T in plain batched tensors: Robin problems on the extended boxes, informed data, basis
    functions, coupling system, reconstruction and Schwarz sweeps."""

    def __init__(self, c, K, h):
        self.c, self.nq, s, l, dev = c, 1 + c["degree"], c["sub"], c["l"], K.device
        nx, ny = c["nx"], c["ny"]
        self.Tx, self.Ty = _trans(c, K, h)
        self.K, self.h = K, h
        self.mx, self.my = -(-nx // s), -(-ny // s)
        S = self.S = self.mx * self.my
        I, J = torch.arange(S, device=dev) % self.mx, torch.arange(S, device=dev) // self.mx
        self.x0, self.y0 = I * s, J * s
        self.robin = torch.stack([I > 0, I < self.mx - 1, J > 0, J < self.my - 1], 1)
        ext, core = self.cells(l), self.cells(0)
        self.ext, self.core = ext, core
        self.dirichlet = Lines(*self.coeffs(ext, False)) if c["sweeps"] else None
        self.outer, self.local = Lines(*self.coeffs(ext, True)), Lines(*self.coeffs(core, True))
        # faces of each subdomain's sides: inside and outside cells, [S, 4, s]
        t = torch.arange(s, device=dev).expand(S, s)
        w, hh = torch.clamp(nx - self.x0, max=s), torch.clamp(ny - self.y0, max=s)
        fx = torch.stack([0 * t, w[:, None] - 1 + 0 * t, t, t], 1)
        fy = torch.stack([t, t, 0 * t, hh[:, None] - 1 + 0 * t], 1)
        self.len = torch.stack([hh, hh, w, w], 1)
        self.on = self.robin[:, :, None] & (t[:, None, :] < self.len[:, :, None])
        step = torch.tensor([[-1, 0], [1, 0], [0, -1], [0, 1]], device=dev)
        self.fx, self.fy = fx, fy
        self.ox, self.oy = fx + step[:, 0, None], fy + step[:, 1, None]
        g = [(self.x0[:, None, None] + a).clamp(0, nx - 1) for a in (fx, self.ox)]
        q = [(self.y0[:, None, None] + a).clamp(0, ny - 1) for a in (fy, self.oy)]
        k_in, k_out = (torch.cat([K[0][q[i], g[i]][:, :2], K[-1][q[i], g[i]][:, 2:]], 1) for i in (0, 1))
        self.tau = 2 * k_in
        self.Tf = 2 * k_in * k_out / (k_in + k_out)
        self.beta = 10.0 * s * h / self.Tf
        self.tr = 1.0 / (1.0 / self.tau + self.beta / h)
        one = torch.ones_like(t[:, None, :] * self.len[:, :, None], dtype=F8)
        lin = 2.0 * (t[:, None, :] + 0.5) / self.len[:, :, None] - 1.0
        self.fn = torch.stack([one, lin][: self.nq], 2) * self.on[:, :, None, :]     # [S, 4, nq, s]
        self.setup()

    def cells(self, l):
        s, dev = self.c["sub"], self.K.device
        a = torch.arange(s + 2 * l, device=dev) - l
        gx, gy = self.x0[:, None] + a, self.y0[:, None] + a
        act = ((gy >= 0) & (gy < self.c["ny"]))[:, :, None] & ((gx >= 0) & (gx < self.c["nx"]))[:, None, :]
        return gx.clamp(0, self.c["nx"] - 1)[:, None, :].expand_as(act), gy.clamp(0, self.c["ny"] - 1)[:, :, None].expand_as(act), act

    def robin_faces(self, box):
        """t_R of the box's outer faces towards cells of the grid, and the transmissibility it replaces."""
        gx, gy, act = box
        nx, ny, out = self.c["nx"], self.c["ny"], []
        for k in range(4):
            dx, dy, ax = ((-1, 0, 0), (1, 0, 0), (0, -1, 1), (0, 1, 1))[k]
            edge = torch.zeros_like(act)
            edge[(slice(None),) + ((slice(None), (0, -1)[k]) if ax == 0 else ((0, -1)[k - 2],))] = True
            inside = ((gx + dx >= 0) & (gx + dx < nx)) if ax == 0 else ((gy + dy >= 0) & (gy + dy < ny))
            Kc = self.K[0] if ax == 0 else self.K[-1]
            ki, ko = Kc[gy, gx], Kc[(gy + dy).clamp(0, ny - 1), (gx + dx).clamp(0, nx - 1)]
            T = 2 * ki * ko / (ki + ko)
            on = edge & inside & act
            out.append((torch.where(on, 1.0 / (1.0 / (2 * ki) + 10.0 * self.c["sub"] / T), 0.0), torch.where(on, T, 0.0)))
        return out

    def coeffs(self, box, robin):
        gx, gy, act = box
        tw, te, ts, tn = self.Tx[gy, gx], self.Tx[gy, gx + 1], self.Ty[gy, gx], self.Ty[gy + 1, gx]
        d = tw + te + ts + tn
        if robin:
            for tr, T in self.robin_faces(box):
                d = d + tr - T
        east = torch.where(act[:, :, :-1] & act[:, :, 1:], te[:, :, :-1], 0.0)
        north = torch.where(act[:, :-1] & act[:, 1:], tn[:, :-1], 0.0)
        return torch.where(act, d, 1.0), east, north

    def at(self, q, fx, fy, l):
        """Values of box functions [S, h, w, R] at local cells (fx, fy) of each subdomain: [S, 4, s, R]."""
        s = torch.arange(self.S, device=q.device)[:, None, None]
        m = q.shape[1] - 1
        return q[s, (fy + l).clamp(0, m), (fx + l).clamp(0, m)]

    def flux(self, q):
        """Flux and face pressure of extended solutions on the subdomain's own faces."""
        qc = self.at(q, self.fx, self.fy, self.c["l"])
        F = self.Tf[..., None] * (qc - self.at(q, self.ox, self.oy, self.c["l"]))
        return F, qc - F / self.tau[..., None]

    def moments(self, F, P):
        """Against the test functions of each side: [S, 4 sides, nq tests, R]."""
        return (torch.einsum("skqt,sktr->skqr", self.fn, F), torch.einsum("skqt,sktr->skqr", self.fn, self.h * P))

    def setup(self):
        c, nq, S, dev = self.c, self.nq, self.S, self.K.device
        gx, gy, act = self.ext
        lo = torch.stack([gy.amin((1, 2))] * 2 + [gx.amin((1, 2))] * 2, 1)
        hi = torch.stack([gy.amax((1, 2))] * 2 + [gx.amax((1, 2))] * 2, 1)
        rhs = []
        for k, (tr, _) in enumerate(self.robin_faces(self.ext)):
            pos = gy if k < 2 else gx
            size = (hi - lo + 1)[:, k, None, None]
            for q in range(nq):
                rhs.append(tr * (2.0 * (pos - lo[:, k, None, None] + 0.5) / size - 1.0 if q else 1.0))
        sol = self.outer.solve(torch.stack(rhs, -1))                      # [S, h, w, 4 nq]
        F, P = self.flux(sol)
        own = torch.repeat_interleave(self.robin, nq, 1)[:, None, None, :]
        phi = torch.where(self.on[..., None] & own, P - self.beta[..., None] * F / self.h, 0.0)
        b = torch.zeros(S, c["sub"], c["sub"], 4 * nq, device=dev, dtype=F8)
        s = torch.arange(S, device=dev)[:, None, None].expand_as(self.fx)
        b.index_put_((s, self.fy, self.fx), torch.where(self.on, self.tr, 0.0)[..., None] * phi, accumulate=True)
        self.psi = self.local.solve(b)
        F = self.tr[..., None] * (self.at(self.psi, self.fx, self.fy, 0) - phi)
        MF, MP = self.moments(F, phi + self.beta[..., None] * F / self.h)
        # coupling rows: flux and pressure of each interface, per test function
        self.idx = (torch.cumsum(self.robin.flatten().long(), 0) - 1).view(S, 4)
        n = int(self.robin.sum()) * nq
        G = torch.zeros(n, n, device=dev, dtype=F8)
        self.rows, e = [], 0
        for a in (0, 1):
            low = torch.nonzero(self.robin[:, 2 * a + 1]).flatten()
            up, r0 = low + (1 if a == 0 else self.mx), 2 * nq * (e + torch.arange(len(low), device=dev))
            e += len(low)
            self.rows.append((a, low, up, r0))
            for t, sign, k in ((low, 1.0, 2 * a + 1), (up, -1.0, 2 * a)):
                for r in range(4):
                    m = self.robin[t, r]
                    for q in range(nq):
                        col = self.idx[t[m], r] * nq + q
                        for qt in range(nq):
                            G.index_put_((r0[m] + qt, col), MF[t[m], k, qt, r * nq + q], accumulate=True)
                            G.index_put_((r0[m] + nq + qt, col), sign * MP[t[m], k, qt, r * nq + q], accumulate=True)
        self.G = torch.linalg.lu_factor(G) if n else None

    def take(self, r, box):
        return torch.where(box[2], r[box[1], box[0]], 0.0)[..., None]

    def put(self, z, boxes, which=None, l=0):
        """Adds each subdomain's own cells of box functions to the grid function z."""
        gx, gy, act = self.core
        m = act if which is None else act & which[:, None, None]
        s = self.c["sub"]
        z[gy[m], gx[m]] += boxes[:, l:l + s, l:l + s, 0][m]
        return z

    def __call__(self, r):
        c, nq = self.c, self.nq
        q0 = self.outer.solve(self.take(r, self.ext))
        F, P = self.flux(q0)
        MF, MP = self.moments(F, P)
        l, s = c["l"], c["sub"]
        z = self.put(torch.zeros_like(r), q0, None, l)
        if self.G is not None:
            g = torch.zeros(self.G[0].shape[0], 1, device=r.device, dtype=F8)
            for a, low, up, r0 in self.rows:
                for qt in range(nq):
                    g[r0 + qt] = -(MF[low, 2 * a + 1, qt] + MF[up, 2 * a, qt])
                    g[r0 + nq + qt] = -(MP[low, 2 * a + 1, qt] - MP[up, 2 * a, qt])
            x = torch.linalg.lu_solve(*self.G, g).flatten().view(-1, nq)
            co = torch.where(self.robin[..., None], x[self.idx.clamp_min(0)], 0.0).reshape(self.S, 1, 1, 4 * nq)
            z = self.put(z, (self.psi * co).sum(-1, keepdim=True))
        colour = (torch.arange(self.S, device=r.device) % self.mx) % 2 + 2 * ((torch.arange(self.S, device=r.device) // self.mx) % 2)
        for _ in range(c["sweeps"]):
            for k in range(4) if c["mult"] else (None,):
                rho = r - _apply(self.Tx, self.Ty, z)
                z = self.put(z, self.dirichlet.solve(self.take(rho, self.ext)), None if k is None else colour == k, l)
        return z


def _pressure(c, Tx, Ty, f, left):
    b = torch.zeros(c["ny"], c["nx"], device=Tx.device, dtype=F8) if f is None else f.clone()
    b[:, 0] += Tx[:, 0] * left
    d = Tx[:, 1:] + Tx[:, :-1] + Ty[1:] + Ty[:-1]
    flip = c["nx"] > c["ny"]       # eliminate along the longer axis
    east, north = Tx[:, 1:-1], Ty[1:-1]
    if flip:
        d, east, north, b = d.t(), north.t(), east.t(), b.t()
    p = Lines(d[None], east[None], north[None]).solve(b[None, ..., None])[0, ..., 0]
    return p.t().contiguous() if flip else p


def exact(case, seed):
    c = _full(case)
    if c["kind"] == "serve":
        out = []
        for i, r in enumerate(_requests(c)):
            K, f, left, _, h = _problem(r, 1000 * seed + i)
            out.append(_pressure(r, *_trans(r, K, h), f, left).flatten().cpu().numpy())
        return out
    K, f, left, v, h = _problem(c, seed)
    Tx, Ty = _trans(c, K, h)
    if c["kind"] == "operator":
        return _apply(Tx, Ty, v.view(c["ny"], c["nx"])).flatten()
    if c["kind"] in ("precond", "setup"):
        return Multiscale(c, K, h)(v.view(c["ny"], c["nx"])).flatten()
    if min(c["nx"], c["ny"]) > 1024:      # the direct elimination takes the fourth power of the width
        return None
    p = _pressure(c, Tx, Ty, f, left)
    if not c["fluxes"]:
        return p.flatten()
    q = torch.nn.functional.pad(p, (1, 1))
    q[:, 0] = left
    ux, uy = Tx * (q[:, :-1] - q[:, 1:]) / h, torch.zeros_like(Ty)
    uy[1:-1] = Ty[1:-1] * (p[:-1] - p[1:]) / h
    return [p.flatten(), ux.flatten(), uy.flatten()]

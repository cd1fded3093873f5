"""Performance cases: what a user of the solver has it do, through the package's public classes.

A case is a dict of plain values.  Kinds:
  step     Solver.step: whole time steps (three RK3 sub-steps each) of one channel or boundary layer
  cfl      Solver.step_cfl: steps at a fixed CFL number, the paper's own way of running
  host     ns_step_host: a step on a state that lives in pinned host memory
  batch    Batch.step: an ensemble of small uneven channels advanced together
  poisson  Solver.poisson: one pressure solve of a given velocity field
  static   ns_poisson_solve_static: the pressure solve that allocates nothing

Inputs follow the recipes of paper_1812_01178_gb300/inputs.py (log-law or laminar or boundary-layer
mean plus fluctuations, projected divergence-free), drawn on the device so that they are quick to
make.  `exact` restates the method in plain torch, in 64 bits.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1812_01178_gb300 import binding as B
from paper_1812_01178_gb300 import inputs as I

GAMMA = (8.0 / 15.0, 5.0 / 12.0, 3.0 / 4.0)
ZETA = (0.0, -17.0 / 60.0, -5.0 / 12.0)
ALPHA = (8.0 / 15.0, 2.0 / 15.0, 1.0 / 3.0)
DEV = "cuda:0"

# nx: lengths 2^a 3^b the x transforms and the x partitions both take; nz: lengths of the z transforms
NX = (16, 24, 32, 48, 64, 72, 96, 128, 144, 192, 256, 288, 384, 512, 768, 1024)
NZ = (8, 16, 24, 32, 48, 64, 72, 96, 128, 144, 192, 216, 256, 288, 384, 512, 648, 1024)


def _case(kind, nx, ny, nz, flow="turbulent", mixed=False, **more):
    return dict({"kind": kind, "nx": nx, "ny": ny, "nz": nz, "flow": flow, "mixed": mixed, "kim_moin": False,
                 "steps": 1, "instances": 1}, **more)


def listed():
    return [
        # a laminar channel at the size of the first validation run: the smallest call, where the
        # 30 launches of a step and the length of each kernel's serial chains count
        dict(_case("step", 64, 64, 32, "laminar"), name="laminar_64x64x32"),
        # the benchmark workload, in both precisions
        dict(_case("step", 256, 192, 256), name="channel_256x192x256"),
        dict(_case("step", 256, 192, 256, mixed=True), name="channel_256x192x256_mixed"),
        # lengths with factors of three and an odd number of rows; no direction fits the tiles
        # evenly; the Kim-Moin pressure update
        dict(_case("step", 144, 101, 216, kim_moin=True), name="channel_144x101x216_kim_moin"),
        # the flat plate with inflow and convective outflow at the size of the paper's runs
        dict(_case("step", 1024, 256, 512, "plate"), name="plate_1024x256x512"),
        dict(_case("step", 1024, 256, 512, "plate", mixed=True), name="plate_1024x256x512_mixed"),
        # a coarse flat plate, as run while a set-up is tried out
        dict(_case("step", 384, 96, 128, "plate"), name="plate_384x96x128"),
        # four steps at CFL 1.0 (dt and all its tables renewed on the device every step)
        dict(_case("cfl", 192, 128, 192, steps=4), name="channel_192x128x192_cfl"),
        # an ensemble of small channels, in both precisions
        dict(_case("batch", 128, 96, 128, "laminar", instances=16), name="ensemble_16"),
        dict(_case("batch", 128, 96, 128, "laminar", mixed=True, instances=16), name="ensemble_16_mixed"),
        # the state on the host, as a coupled code has it: copies in, one step, copies out
        dict(_case("host", 256, 192, 256), name="channel_256x192x256_host"),
        # one pressure solve without an allocation, inside another program's time loop
        dict(_case("static", 96, 64, 96), name="poisson_static_96x64x96"),
    ]


def _cells(case):
    if case["kind"] == "batch":
        return sum(math.prod(s) for s in _ensemble_sizes(case))
    return case["nx"] * case["ny"] * case["nz"]


def draw(rng):
    kind = rng.choice(("step", "step", "step", "step", "cfl", "batch", "poisson", "static", "host"))
    flow = rng.choice(("turbulent", "laminar", "plate")) if kind == "step" else "turbulent"
    mixed = rng.random() < 0.3 and kind in ("step", "cfl", "batch", "poisson")
    if kind == "batch":
        return _case("batch", 128, 96, 128, "laminar", mixed, instances=rng.randint(3, 24))
    # sizes spread over the logarithm of the cell count, then over the shapes that give about it
    top = {"step": 6.4e7, "cfl": 1.2e7, "poisson": 3.2e7, "static": 1.2e6, "host": 8e6}[kind]
    want = math.exp(rng.uniform(math.log(3e4), math.log(top)))
    while True:
        nx, nz = rng.choice(NX), rng.choice(NZ)
        ny = rng.randint(4, 384)
        if 0.6 * want < nx * ny * nz < 1.4 * want and max(nx, ny, nz) <= 24 * min(nx, ny, nz):
            break
    return _case(kind, nx, ny, nz, flow, mixed, kim_moin=kind == "step" and rng.random() < 0.25,
                 steps=rng.randint(1, 4) if kind == "cfl" else 1)


# ------------------------------------------------------------------------------ inputs
def _ensemble_sizes(case):
    """Sizes of the ensemble's instances: the recipe of inputs.ensemble."""
    out = []
    for i in range(case["instances"]):
        r = I.uniform01(1812 + i, 3)
        out.append(((32, 64, case["nx"])[int(r[0] * 3)], (32, 48, 64, case["ny"])[int(r[2] * 4)],
                    (32, 64, case["nz"])[int(r[1] * 3)]))
    return out


def _make(case, seed):
    """(inputs.Case, u, v, w, p, boundary planes or None): the raw fields, not yet projected."""
    nx, ny, nz, flow = case["nx"], case["ny"], case["nz"], case["flow"]
    g = torch.Generator(device=DEV).manual_seed(int(seed) * 7919 + 17)

    def noise(*shape):
        return torch.randn(shape, generator=g, dtype=torch.float64, device=DEV)

    def col(a):
        return torch.as_tensor(a, dtype=torch.float64, device=DEV)[None, :, None]

    bl = None
    if flow == "plate":
        c = I.boundary_layer_case(nx, ny, nz)
        yc = 0.5 * (c.yf[:-1] + c.yf[1:])
        prof, amp = np.tanh(2.0 * yc), 1e-2
        u = col(prof) + amp * noise(nz, ny, nx)
        v, w = amp * noise(nz, ny + 1, nx), amp * noise(nz, ny, nx)
        v[:, 0] = v[:, ny] = 0.0
        v_in = amp * noise(nz, ny + 1)
        v_in[:, 0] = v_in[:, ny] = 0.0
        bl = {"u_out": u[:, :, -1].clone(), "v_in": v_in, "v_out": v[:, :, -1].clone(),
              "w_in": amp * noise(nz, ny), "w_out": w[:, :, -1].clone()}
    elif flow == "laminar":
        re, amp = 2000.0, 1e-3
        c = I.Case("laminar", nx, ny, nz, 2 * math.pi, math.pi, I.channel_faces(ny, 2.0), re=re, fx=3.0 / re)
        yc = 0.5 * (c.yf[:-1] + c.yf[1:])
        u = col(1.5 * (1.0 - yc ** 2)) + amp * noise(nz, ny, nx)
        v, w = amp * noise(nz, ny + 1, nx), amp * noise(nz, ny, nx)
        v[:, 0] = v[:, ny] = 0.0
    else:
        re = 395.0
        c = I.Case("turbulent", nx, ny, nz, 2 * math.pi, math.pi, I.channel_faces(ny, 2.0), re=re, fx=1.0)
        yc = 0.5 * (c.yf[:-1] + c.yf[1:])
        mean = I.loglaw_mean((1.0 - np.abs(yc)) * re)
        meanf = I.loglaw_mean((1.0 - np.abs(c.yf)) * re)
        u = col(mean) + col(0.1 * mean) * noise(nz, ny, nx)
        v, w = col(0.1 * meanf) * noise(nz, ny + 1, nx), col(0.1 * mean) * noise(nz, ny, nx)
        v[:, 0] = v[:, ny] = 0.0
    # a smooth pressure of the size of the velocity fluctuations squared
    ph = torch.rand(4, generator=g, dtype=torch.float64, device=DEV).tolist()
    xs, zs = (torch.arange(n, dtype=torch.float64, device=DEV) / n for n in (nx, nz))
    px = torch.cos(2 * math.pi * (3 * xs + ph[0])) + torch.sin(2 * math.pi * (xs + ph[1]))
    pz = torch.cos(2 * math.pi * (2 * zs + ph[2])) + torch.sin(2 * math.pi * (zs + ph[3]))
    ys = torch.cos(math.pi * torch.arange(ny, dtype=torch.float64, device=DEV) / ny)
    scale = {"plate": 1e-3, "laminar": 1e-4, "turbulent": 1.0}[flow]
    p = scale * pz[:, None, None] * ys[None, :, None] * px[None, None, :]
    c.precision = B.NS_MIXED if case["mixed"] else B.NS_FP64
    c.pressure_update = B.NS_PRESSURE_KIM_MOIN if case["kim_moin"] else B.NS_PRESSURE_DELTA
    if case["kind"] == "batch":
        c.dt = 2e-3  # one time step for the whole ensemble
    else:
        c.dt = 0.5 / _rate(c, u, v, w)
    return c, u, v, w, p.contiguous(), bl


def _members(case, seed):
    """The instances of an ensemble, as (case dict, seed) pairs."""
    return [(dict(case, nx=s[0], ny=s[1], nz=s[2]), seed * 1000 + q) for q, s in enumerate(_ensemble_sizes(case))]


def prepare(case, seed):
    kind = case["kind"]
    if kind == "batch":
        made = [_make(c, s) for c, s in _members(case, seed)]
        b = B.Batch([m[0] for m in made], [[t.cpu().numpy() for t in m[1:5]] for m in made], device=DEV)
        b.make_divergence_free()
        b.sync()
        return {"kind": kind, "batch": b}
    c, u, v, w, p, bl = _make(case, seed)
    if kind == "static":
        return {"kind": kind, "cfg": B.make_config(c), "u": u, "v": v, "w": w, "phi": torch.empty_like(p),
                "stream": torch.cuda.current_stream().cuda_stream}
    s = B.Solver(c, u, v, w, p, device=DEV, bl=bl)
    if kind != "poisson":
        s.make_divergence_free()
    s.sync()
    st = {"kind": kind, "solver": s, "steps": case["steps"]}
    if kind == "host":
        st["host"] = [t.cpu().pin_memory() for t in (s.u, s.v, s.w, s.p)]
        st["arrays"] = [t.numpy() for t in st["host"]]
    return st


def run(st):
    kind = st["kind"]
    if kind == "batch":
        b = st["batch"]
        b.step(1)
        return [t for m in b.t for t in m]
    if kind == "static":
        B.ns_poisson_solve_static(st["cfg"], st["u"].data_ptr(), st["v"].data_ptr(), st["w"].data_ptr(),
                                  st["phi"].data_ptr(), 0, st["stream"])
        return {"phi": st["phi"]}
    s = st["solver"]
    if kind == "poisson":
        s.poisson(0)
        return {"phi": s.buffer(B.NS_BUF_PHI)}
    if kind == "host":
        B.ns_step_host(s.ctx, *st["arrays"], 1)
        return dict(zip("uvwp", st["arrays"]))
    out = {"u": s.u, "v": s.v, "w": s.w, "p": s.p}
    if kind == "cfl":
        out["dt"] = np.array(s.step_cfl(st["steps"], 1.0))
    else:
        s.step(st["steps"])
    for q in ("u_out", "v_out", "w_out"):
        if s.bl:
            out[q] = s.bl[q]
    return out


def work(case):
    """State in and out once (u, v, w, p), and the arithmetic of the method: per cell and sub-step
    150 for the right-hand side, 5 per point and line solve (three components, three directions), the
    transforms at 5 N log2 N, 10 per complex point of the y solve, 24 for divergence and projection."""
    cells = _cells(case)
    members = _ensemble_sizes(case) if case["kind"] == "batch" else [(case["nx"], case["ny"], case["nz"])]
    poisson = sum(math.prod(s) * (5 * math.log2(s[2]) + 5 * math.log2(s[0]) + 5 + 9) for s in members)
    if case["kind"] in ("poisson", "static"):
        return {"bytes": 8 * 4 * cells, "flops": poisson}
    n = 3 * case["steps"]
    return {"bytes": 8 * 8 * cells, "flops": n * (cells * (150 + 45 + 3 + 15) + poisson)}


# ------------------------------------------------------------------------------ the method in 64 bits
def _up(f, d):
    return torch.roll(f, -1, d)


def _dn(f, d):
    return torch.roll(f, 1, d)


def _rate(c, u, v, w):
    dy = torch.as_tensor(np.diff(c.yf), device=u.device)[None, :, None]
    vc = 0.5 * (v[:, :-1] + v[:, 1:])
    return float((u.abs() / (c.lx / c.nx) + vc.abs() / dy + w.abs() / (c.lz / c.nz)).max())


class _Method:
    """One flow in plain torch: staggered second-order differences, RK3 / Crank-Nicolson fractional
    steps, exact line solves, the pressure by transforms in x and z and a line solve in y."""

    def __init__(self, c, device):
        self.c, self.plate = c, c.bc_x == 1
        self.dx, self.dz = c.lx / c.nx, c.lz / c.nz
        yf = np.asarray(c.yf, dtype=np.float64)
        yc, dy = 0.5 * (yf[:-1] + yf[1:]), np.diff(yf)
        hc = np.diff(yc)
        hm, hp = np.concatenate([[yc[0] - yf[0]], hc]), np.concatenate([hc, [yf[-1] - yc[-1]]])
        lo, hi = 2.0 / (hm * (hm + hp)), 2.0 / (hp * (hm + hp))
        if c.bc_ytop == 1:
            hi[-1] = 0.0
        t = lambda a: torch.as_tensor(a, dtype=torch.float64, device=device)
        self.dy, self.hc = t(dy)[None, :, None], t(hc)[None, :, None]
        self.whi = t((yf[1:-1] - yc[:-1]) / hc)[None, :, None]
        self.centre, self.face = (t(lo), t(hi)), (t(2.0 / (dy[:-1] * (dy[:-1] + dy[1:]))), t(2.0 / (dy[1:] * (dy[:-1] + dy[1:]))))
        self.pa, self.pc = t(np.concatenate([[0.0], 1.0 / (dy[1:] * hc)])), t(np.concatenate([1.0 / (dy[:-1] * hc), [0.0]]))
        self.area = (yf[-1] - yf[0]) * c.lz
        self.device = device

    # ---- values next to a point in x
    def ux(self, u, bl):
        return torch.cat([u[:, :, 1:], bl["u_out"][:, :, None]], 2) if self.plate else _up(u, 2)

    def cx(self, f, bl, q):
        return torch.cat([f[:, :, 1:], (2.0 * bl[q + "_out"] - f[:, :, -1])[:, :, None]], 2) if self.plate else _up(f, 2)

    def xm(self, f, bl, q=None):
        if not self.plate:
            return _dn(f, 2)
        first = torch.zeros_like(f[:, :, :1]) if q is None else (2.0 * bl[q + "_in"] - f[:, :, 0])[:, :, None]
        return torch.cat([first, f[:, :, :-1]], 2)

    def yface(self, f):
        out = torch.zeros((f.shape[0], self.c.ny + 1, f.shape[2]), dtype=f.dtype, device=f.device)
        out[:, 1:-1] = (1.0 - self.whi) * f[:, :-1] + self.whi * f[:, 1:]
        return out

    def dyy(self, f, rows, inner):
        a, cc = (q[None, :, None] for q in rows)
        out = torch.zeros_like(f)
        if inner:
            out[:, 1:-1] = a * f[:, :-2] - (a + cc) * f[:, 1:-1] + cc * f[:, 2:]
        else:
            out -= (a + cc) * f
            out[:, 1:] += a[:, 1:] * f[:, :-1]
            out[:, :-1] += cc[:, :-1] * f[:, 1:]
        return out

    def convection(self, u, v, w, bl):
        dx, dz, dy, hc = self.dx, self.dz, self.dy, self.hc
        uc = 0.5 * (u + self.ux(u, bl))
        fuv = self.yface(u) * (0.5 * (self.xm(v, bl, "v") + v))
        fuw = 0.5 * (_dn(u, 0) + u) * (0.5 * (self.xm(w, bl, "w") + w))
        if self.plate:
            uo = bl["u_out"][:, :, None]
            fuv_n = torch.cat([fuv[:, :, 1:], self.yface(uo) * bl["v_out"][:, :, None]], 2)
            fuw_n = torch.cat([fuw[:, :, 1:], 0.5 * (_dn(uo, 0) + uo) * bl["w_out"][:, :, None]], 2)
        else:
            fuv_n, fuw_n = _up(fuv, 2), _up(fuw, 2)
        nu = (uc * uc - self.xm(uc, bl) ** 2) / dx + (fuv[:, 1:] - fuv[:, :-1]) / dy + (_up(fuw, 0) - fuw) / dz
        if self.plate:
            nu[:, :, 0] = 0.0
        vc = 0.5 * (v[:, :-1] + v[:, 1:])
        fvw = 0.5 * (_dn(v, 0) + v) * self.yface(w)
        nv = (fuv_n - fuv) / dx + (_up(fvw, 0) - fvw) / dz
        nv[:, 1:-1] += (vc[:, 1:] ** 2 - vc[:, :-1] ** 2) / hc
        nv[:, 0] = nv[:, -1] = 0.0
        wc = 0.5 * (w + _up(w, 0))
        nw = (fuw_n - fuw) / dx + (fvw[:, 1:] - fvw[:, :-1]) / dy + (wc * wc - _dn(wc, 0) ** 2) / dz
        return [nu, nv, nw]

    def gradient(self, p):
        gx = (p - _dn(p, 2)) / self.dx
        if self.plate:
            gx[:, :, 0] = 0.0
        gy = torch.zeros((p.shape[0], self.c.ny + 1, p.shape[2]), dtype=p.dtype, device=p.device)
        gy[:, 1:-1] = (p[:, 1:] - p[:, :-1]) / self.hc
        return [gx, gy, (p - _dn(p, 0)) / self.dz]

    def divergence(self, u, v, w, bl):
        return (self.ux(u, bl) - u) / self.dx + (v[:, 1:] - v[:, :-1]) / self.dy + (_up(w, 0) - w) / self.dz

    def viscous(self, f, q, up, dn):
        lap = (up - 2.0 * f + dn) / self.dx ** 2 + (_up(f, 0) - 2.0 * f + _dn(f, 0)) / self.dz ** 2
        return lap + (self.dyy(f, self.face, True) if q == 1 else self.dyy(f, self.centre, False))

    # ---- line solves
    @staticmethod
    def thomas(a, b, c, d):
        """Rows along dim 0; a, b, c 1-D lists of numbers or tensors that broadcast against d[0]."""
        n = d.shape[0]
        x = torch.empty_like(d)
        cp = [None] * n
        piv = b[0]
        cp[0], x[0] = c[0] / piv, d[0] / piv
        for j in range(1, n):
            piv = b[j] - a[j] * cp[j - 1]
            cp[j] = c[j] / piv
            x[j] = (d[j] - a[j] * x[j - 1]) / piv
        for j in range(n - 2, -1, -1):
            x[j] -= cp[j] * x[j + 1]
        return x

    @staticmethod
    def circulant(f, dim, r):
        n = f.shape[dim]
        k = torch.arange(n // 2 + 1, dtype=torch.float64, device=f.device)
        lam = 1.0 + 2.0 * r * (1.0 - torch.cos(2.0 * math.pi * k / n))
        lam = lam.reshape([-1 if q == dim else 1 for q in range(3)])
        return torch.fft.irfft(torch.fft.rfft(f, dim=dim) / lam, n=n, dim=dim)

    def sweep_x(self, f, q, beta, inc):
        r = beta / self.dx ** 2
        if not self.plate:
            return self.circulant(f, 2, r)
        n = self.c.nx
        a, b, cc = [-r] * n, [1.0 + 2.0 * r] * n, [-r] * n
        a[0] = cc[-1] = 0.0
        d = f.permute(2, 0, 1).contiguous()
        if q == 0:
            b[0], cc[0] = 1.0, 0.0
            d[-1] += r * inc
        else:
            b[0] = b[-1] = 1.0 + 3.0 * r
            d[-1] += 2.0 * r * inc
        return self.thomas(a, b, cc, d).permute(1, 2, 0).contiguous()

    def sweep_y(self, f, q, beta):
        lo, hi = (t.tolist() for t in (self.face if q == 1 else self.centre))
        a, b, cc = [-beta * s for s in lo], [1.0 + beta * (s + t) for s, t in zip(lo, hi)], [-beta * t for t in hi]
        out = torch.zeros_like(f)
        inner = f[:, 1:-1] if q == 1 else f
        x = self.thomas(a, b, cc, inner.permute(1, 0, 2).contiguous()).permute(1, 0, 2)
        if q == 1:
            out[:, 1:-1] = x
        else:
            out.copy_(x)
        return out

    def poisson(self, b):
        c = self.c
        nx, nz = c.nx, c.nz
        kx = torch.arange(nx, dtype=torch.float64, device=b.device)
        kz = torch.arange(nz // 2 + 1, dtype=torch.float64, device=b.device)
        lz = (2.0 / self.dz ** 2) * (1.0 - torch.cos(2.0 * math.pi * kz / nz))
        if self.plate:  # cosine transform: the even extension's Fourier transform
            lx = (2.0 / self.dx ** 2) * (1.0 - torch.cos(math.pi * kx / nx))
            half = torch.polar(torch.ones_like(kx), -math.pi * kx / (2 * nx))
            hat = 0.5 * (torch.fft.fft(torch.cat([b, b.flip(2)], 2), dim=2)[:, :, :nx] * half).real
        else:
            lx = (2.0 / self.dx ** 2) * (1.0 - torch.cos(2.0 * math.pi * kx / nx))
            hat = b
        hat = torch.fft.rfft(hat, dim=0)
        if not self.plate:
            hat = torch.fft.fft(hat, dim=2)
        lam = (lz[:, None] + lx[None, :])
        d = hat.permute(1, 0, 2).contiguous()
        del hat
        d[0, 0, 0] = 0.0
        pa, pc = self.pa.tolist(), self.pc.tolist()
        diag = [-(s + t) - lam for s, t in zip(pa, pc)]
        up = [torch.full_like(lam, t) for t in pc]
        diag[0][0, 0], up[0][0, 0] = 1.0, 0.0
        ph = self.thomas(pa, diag, up, d).permute(1, 0, 2)
        del d, diag, up
        if not self.plate:
            return torch.fft.irfft(torch.fft.ifft(ph, dim=2), n=nz, dim=0).contiguous()
        ph = torch.fft.irfft(ph, n=nz, dim=0)
        # DCT-III: x_i = (X_0 + 2 sum X_l cos(pi l (2 i + 1) / (2 nx))) / nx, as one transform of 2 nx
        ext = torch.zeros((ph.shape[0], ph.shape[1], 2 * nx), dtype=torch.complex128, device=b.device)
        ext[:, :, :nx] = ph * half.conj() * 2.0
        ext[:, :, 0] *= 0.5
        return (torch.fft.ifft(ext, dim=2).real[:, :, :nx] * 2.0).contiguous()

    # ---- steps
    def flux_correct(self, u, bl):
        w = self.dy[0, :, 0][None, :] * self.dz
        bl["u_out"] = bl["u_out"] + ((u[:, :, 0] * w).sum() - (bl["u_out"] * w).sum()) / self.area

    def projected(self, u, v, w, bl):
        if self.plate:
            bl = dict(bl)
            self.flux_correct(u, bl)
        g = self.gradient(self.poisson(self.divergence(u, v, w, bl)))
        return [u - g[0], v - g[1], w - g[2]], bl

    def substep(self, vel, p, bl, prev, k, dt):
        c, plate = self.c, self.plate
        u, v, w = vel
        n = self.convection(u, v, w, bl)
        g = self.gradient(p)
        beta = 0.5 * ALPHA[k] * dt / c.re
        new, inc = dict(bl or {}), [None] * 3
        if plate:
            for q, (name, h) in enumerate((("u", self.dx), ("v", 0.5 * self.dx), ("w", 0.5 * self.dx))):
                old = bl[name + "_out"]
                t = old - ALPHA[k] * dt * c.u_conv * (old - vel[q][:, :, -1]) / h
                if q == 1:
                    t[:, 0] = t[:, -1] = 0.0
                new[name + "_out"], inc[q] = t, t - old
        star = []
        for q, f in enumerate(vel):
            up = self.ux(f, bl) if q == 0 else self.cx(f, bl, "uvw"[q])
            dn = self.xm(f, bl, None if q == 0 else "uvw"[q])
            r = -GAMMA[k] * n[q] - ALPHA[k] * g[q] + (ALPHA[k] / c.re) * self.viscous(f, q, up, dn)
            if k:
                r -= ZETA[k] * prev[q]
            if q == 0:
                r += ALPHA[k] * c.fx
                if plate:
                    r[:, :, 0] = 0.0
            if q == 1:
                r[:, 0] = r[:, -1] = 0.0
            r = self.sweep_y(self.sweep_x(dt * r, q, beta, inc[q]), q, beta)
            star.append(f + self.circulant(r, 0, beta / self.dz ** 2))
        del g
        if plate:
            self.flux_correct(u, new)
        s = ALPHA[k] * dt
        phi = self.poisson(self.divergence(*star, new) / s)
        g = self.gradient(phi)
        vel = [a - s * b for a, b in zip(star, g)]
        p = p + phi
        if c.pressure_update == B.NS_PRESSURE_KIM_MOIN:
            p = p - beta * self.divergence(*g, {"u_out": torch.zeros_like(phi[:, :, 0])})
        return vel, p, new, n

    def step(self, vel, p, bl, dt):
        n = None
        for k in range(3):
            vel, p, bl, n = self.substep(vel, p, bl, n, k, dt)
        return vel, p, bl


def exact(case, seed):
    kind = case["kind"]
    if kind == "batch":
        out = []
        for c, s in _members(case, seed):
            r = _exact_step(_make(c, s), 1, None)
            out += [r[q] for q in "uvwp"]
        return out
    made = _make(case, seed)
    if kind in ("poisson", "static"):
        c, u, v, w, _, bl = made
        m = _Method(c, u.device)
        return {"phi": m.poisson(m.divergence(u, v, w, bl) / (ALPHA[0] * c.dt))}
    return _exact_step(made, case["steps"], 1.0 if kind == "cfl" else None)


def _exact_step(made, steps, cfl):
    c, u, v, w, p, bl = made
    m = _Method(c, u.device)
    vel, bl = m.projected(u, v, w, bl)
    del u, v, w
    dts = []
    for _ in range(steps):
        dts.append(cfl / _rate(c, *vel) if cfl else c.dt)
        vel, p, bl = m.step(vel, p, bl, dts[-1])
    out = dict(zip("uvwp", (*vel, p)))
    if cfl:
        out["dt"] = np.array(dts)
    if c.bc_x == 1:
        out.update({q: bl[q] for q in ("u_out", "v_out", "w_out")})
    return out

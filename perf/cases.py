"""The work that users of this package have it do, as cases to be timed and compared.

A pass is what one iteration of a user's time loop does: it steps a prepared simulation (or a batch of them)
through the public entry points and reads a snapshot of its state into device memory. The snapshot holds what a run
is done for (alpha, the pressure, the velocity, the fluxes that carry alpha on), in FP64 for an FP64 run and in FP32
for a mixed-precision one, whose fields are FP32. Geometry, fluids, time steps and solver tolerances are those of the
package's own generators and benchmark: dt_cr = 0.99 of the Brackbill limit, dt_vd = sub dt_cr, `sub` relaxation
sub-steps (fewer where the exit test ends them).

`exact` restates the method in plain FP64 torch (dense arrays, whole-grid operations, Jacobi-preconditioned conjugate
gradients to 1e-14 (1e-12 beside mixed precision) or a dense factorisation), for the sizes where that takes seconds.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2105_10576_gb300 import inputs
from paper_2105_10576_gb300 import oscar as ox
from paper_2105_10576_gb300.batch import Batch

FP64, MIXED = inputs.PREC_FP64, inputs.PREC_MIXED


def _case(geom, step, nx, ny, nz, prec, sub=0, inst=1, name=None):
    c = dict(geom=geom, step=step, nx=nx, ny=ny, nz=nz, prec=prec, sub=sub, inst=inst)
    return dict(c, name=name) if name else c


def listed():
    return [
        # the smallest call: one standard time step of the 128x16 bubble channel (a run takes 2000 of them)
        _case("bubble", "standard", 128, 16, 1, "f64", name="bubble_std_128x16_f64"),
        # the same channel as operator splitting runs it, in both precisions
        _case("bubble", "oscar", 128, 16, 1, "f64", sub=10, name="bubble_128x16_f64"),
        _case("bubble", "oscar", 128, 16, 1, "mixed", sub=10, name="bubble_128x16_mixed"),
        # the paper's first benchmark (bubble and film in a 600x100 um channel, 1 um cells), in FP64
        _case("film", "oscar", 600, 100, 1, "f64", sub=4, name="film_600x100_f64"),
        # the largest grid of the batched sweep on its own: an ordinary 2D run
        _case("bubble", "oscar", 1024, 128, 1, "mixed", sub=4, name="bubble_1024x128_mixed"),
        # the batched sweep: independent channels of uneven size, stepped together
        _case("bubble", "batch", 1024, 128, 1, "mixed", sub=4, inst=10, name="batch_10_mixed"),
        # standard stepping of a rough porous medium whose sizes divide by nothing
        _case("micromodel", "standard", 509, 253, 1, "mixed", name="micromodel_std_509x253_mixed"),
        # the oil-wet micromodel at full size; the exit test on E_k ends the relaxation
        _case("micromodel", "oscar", 2048, 1024, 1, "mixed", sub=4, name="micromodel_2048x1024_mixed"),
        # a served request's small 3D channel, ragged
        _case("constriction", "oscar", 97, 51, 45, "mixed", sub=6, name="constriction_97x51x45_mixed"),
        # the headline: the CO2 slug in the 3D constriction
        _case("constriction", "oscar", 256, 64, 64, "mixed", sub=6, name="constriction_256x64x64_mixed"),
        # the FP64 run that mixed precision is checked against
        _case("constriction", "oscar", 128, 32, 32, "f64", sub=3, name="constriction_128x32x32_f64"),
        # the largest grid that is served
        _case("constriction", "oscar", 256, 128, 128, "mixed", sub=2, name="constriction_256x128x128_mixed"),
    ]


def draw(rng):
    def size(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["bubble", "bubble", "film", "micromodel", "constriction", "constriction", "batch"])
    step = rng.choice(["oscar", "oscar", "standard"])
    prec = rng.choice(["mixed", "mixed", "f64"])
    if kind == "batch":
        ny = size(16, 128)
        return _case("bubble", "batch", 8 * ny + rng.randrange(-3, 4), ny, 1, "mixed", sub=rng.randint(2, 4),
                     inst=rng.randint(3, 10))
    if kind == "bubble":
        ny = size(16, 128)
        nx = 8 * ny + rng.randrange(-3, 4)
        if prec == "f64":
            ny, nx = min(ny, 64), min(nx, 512)
        return _case("bubble", step, nx, ny, 1, prec, sub=rng.randint(3, 10) if step == "oscar" else 0)
    if kind == "film":
        ny = size(20, 100)
        return _case("film", step, 6 * ny, ny, 1, prec, sub=rng.randint(2, 4) if step == "oscar" else 0)
    if kind == "micromodel":
        nx = size(400, 2000)
        return _case("micromodel", step, nx, nx // 2 + rng.randrange(-5, 6), 1, "mixed",
                     sub=rng.randint(2, 4) if step == "oscar" else 0)
    ny = size(24, 100)
    nz = ny + rng.randrange(-3, 4)
    nx = rng.randint(48, 256)
    if prec == "f64":
        nx, ny, nz = min(nx, 120), min(ny, 32), min(nz, 33)
    return _case("constriction", step, nx, ny, nz, prec, sub=rng.randint(2, 6) if step == "oscar" else 0)


# ----------------------------------------------------------------------------
# inputs
# ----------------------------------------------------------------------------
_solids: dict = {}


def _micromodel(nx, ny, rng):
    """Discs on a jittered hexagonal lattice over 4x2 mm (porosity about 0.6, gaps of at least 30 um; the rock of a
    grid size is the same for every run on it), the invading water at x below a seeded front, the fluids of
    inputs.micromodel_2d."""
    Lx, Ly = 4e-3, 2e-3
    hx, hy = Lx / nx, Ly / ny
    if (nx, ny) not in _solids:
        rock = np.random.default_rng(nx * 100003 + ny)
        x = (np.arange(nx) + 0.5) * hx
        y = (np.arange(ny) + 0.5) * hy
        solid = np.zeros((ny, nx), np.uint8)
        pitch = 230e-6
        row = 0
        cy = 0.5 * pitch
        while cy < Ly - 0.45 * pitch:
            cx = 0.15e-3 + 0.5 * pitch + 0.5 * pitch * (row % 2)
            while cx < Lx - 0.15e-3 - 0.5 * pitch:
                r = rock.uniform(55e-6, 90e-6)
                px, py = cx + rock.uniform(-10e-6, 10e-6), cy + rock.uniform(-10e-6, 10e-6)
                i0, i1 = max(int((px - r) / hx) - 1, 0), min(int((px + r) / hx) + 2, nx)
                j0, j1 = max(int((py - r) / hy) - 1, 0), min(int((py + r) / hy) + 2, ny)
                solid[j0:j1, i0:i1] |= ((x[None, i0:i1] - px) ** 2 + (y[j0:j1, None] - py) ** 2 <= r * r).astype(np.uint8)
                cx += pitch
            cy += pitch * math.sqrt(3.0) / 2
            row += 1
        _solids[nx, ny] = inputs.keep_outlet_connected(solid)
    solid = _solids[nx, ny]
    sigma, mu_w = 0.035, 1e-3
    Ca = 10.0 ** rng.uniform(-6, -4)
    p = inputs.default_params(dim=2, nx=nx, ny=ny, nz=1, hx=hx, hy=hy, hz=hx, rho1=1000.0, rho2=850.0, mu1=mu_w,
                              mu2=5e-3, sigma=sigma, theta_deg=150.0, U_inlet=Ca * sigma / mu_w, alpha_inlet=1.0)
    front = rng.uniform(0.2, 0.5) * Lx
    edge = np.clip((front - np.arange(nx) * hx) / hx, 0.0, 1.0)
    alpha0 = np.where(solid == 1, 0.0, np.broadcast_to(edge[None, :], (ny, nx)))
    return inputs.Case("micromodel", p, solid, alpha0, {})


def _make(case, seed, q=0):
    """Instance q of a case: the geometry of its generator, its fluids' speed, positions and lengths from the seed."""
    rng = np.random.default_rng([seed, q])
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    mixed = case["prec"] == "mixed"
    over = dict(precision=MIXED if mixed else FP64, cg_rtol=1e-8 if mixed else 1e-13)
    if case["geom"] == "bubble":
        if case["step"] == "batch":   # instance q on the grid, or on a half, a quarter, an eighth of it
            nx, ny = max(nx >> (q % 4), 16), max(ny >> (q % 4), 4)
        return inputs.channel_bubble_2d(nx=nx, ny=ny, Ca=10.0 ** rng.uniform(-6, -3),
                                        bubble_len=rng.uniform(2.0, 5.0) * 100e-6, conv_tol=1e-6,
                                        bubble_x=rng.uniform(350e-6, 450e-6), **over)
    if case["geom"] == "film":
        over["cg_rtol"] = 1e-8 if mixed else 1e-10
        return inputs.bubble_film_2d(Ca=10.0 ** rng.uniform(-3, -1.5), h=600e-6 / nx, bubble_len=rng.uniform(150e-6, 250e-6),
                                     bubble_x0=rng.uniform(20e-6, 80e-6), **over)
    if case["geom"] == "micromodel":
        c = _micromodel(nx, ny, rng)
        c.params.update(over)
        return c
    return inputs.constricted_channel_3d(nx=nx, ny=ny, nz=nz, Ca=10.0 ** rng.uniform(-6, -4), throat=0.30,
                                         slug_frac=rng.uniform(0.3, 0.5), **over)


def _steps(p, sub):
    """(dt_vd, dt_cr): 0.99 of the Brackbill limit per sub-step, `sub` sub-steps to a drag step."""
    h = min(p["hx"], p["hy"], p["hz"] if p["dim"] == 3 else p["hx"])
    dt = 0.99 * math.sqrt(0.5 * (p["rho1"] + p["rho2"]) * h ** 3 / (2.0 * math.pi * p["sigma"]))
    return max(sub, 1) * dt, dt


def _snapshot_fields(p, step):
    phi = ox.FIELD_PHI_VD if step == "standard" else ox.FIELD_PHI_CR
    d = range(p["dim"])
    return ([("alpha", ox.FIELD_ALPHA), ("p", ox.FIELD_P)] + [("u" + "xyz"[a], ox.FIELD_U + a) for a in d]
            + [("phi" + "xyz"[a], phi + a) for a in d])


class _Sim:
    """A simulation as a user holds it: the handle on a stream of its own, the time steps, the snapshot's buffers."""

    def __init__(self, case, seed, q):
        c = _make(case, seed, q)
        self.p = c.params
        self.stream = torch.cuda.Stream()
        self.sim = ox.Oscar(self.p, c.solid, c.alpha0, self.stream.cuda_stream)
        self.dt_vd, self.dt_cr = _steps(self.p, case["sub"])
        self.out, self.buf = {}, {}
        with torch.cuda.stream(self.stream):
            for name, which in _snapshot_fields(self.p, case["step"]):
                n, shape = self.sim._len_shape(which)
                f64 = torch.empty(shape, dtype=torch.float64, device="cuda")
                self.buf[name] = (which, n, f64)
                self.out[name] = f64 if self.p["precision"] == FP64 else torch.empty(shape, dtype=torch.float32, device="cuda")

    def snapshot(self):
        with torch.cuda.stream(self.stream):
            for name, (which, n, f64) in self.buf.items():
                self.sim.field_device(which, f64.data_ptr(), n)
                if self.out[name] is not f64:
                    self.out[name].copy_(f64)
        torch.cuda.current_stream().wait_stream(self.stream)
        return dict(self.out)


def prepare(case, seed):
    sims = [_Sim(case, seed, q) for q in range(case["inst"])]
    return dict(case=case, sims=sims, batch=Batch([s.sim for s in sims]) if case["step"] == "batch" else None)


def run(state):
    case, sims = state["case"], state["sims"]
    if case["step"] == "batch":
        state["batch"].step([s.dt_vd for s in sims], [s.dt_cr for s in sims], [case["sub"]] * len(sims))
        return [s.snapshot() for s in sims]
    s = sims[0]
    if case["step"] == "standard":
        s.sim.standard_step(s.dt_cr)
        return s.snapshot()
    s.sim.drag_step(s.dt_vd)
    s.sim.relax(s.dt_cr, case["sub"])
    return s.snapshot()


def work(case):
    """Per cell and step (a standard or drag step, or a relaxation sub-step): the state read and written once (alpha,
    velocity, both fluxes, pressure, the cell's face types), and the operations of the transport, the interface, three
    momentum predictions and, per pressure solve, one application of the operator."""
    dim = 3 if case["nz"] > 1 else 2
    e = 8 if case["prec"] == "f64" else 4
    steps = 1 + case["sub"] if case["step"] != "standard" else 1
    cells = 0
    for q in range(case["inst"]):
        s = q % 4 if case["step"] == "batch" else 0
        cells += max(case["nx"] >> s, 1) * max(case["ny"] >> s, 1) * case["nz"]
    per_cell = e * (2 + 2 * dim + 3 * dim) + 16 + 4
    snap = (e if case["prec"] == "f64" else 4) * (2 + 2 * dim)
    flops = 60 * dim + 40 * dim + 3 * (25 * dim * dim + 12 * dim)
    return {"bytes": cells * (steps * per_cell + snap), "flops": cells * steps * flops}


# ----------------------------------------------------------------------------
# the method in plain FP64 torch
# ----------------------------------------------------------------------------
class _Exact:
    """Arrays have the grid's shape (x the last axis); a face array of direction a has one more entry along it."""

    def __init__(self, p, solid, alpha0, device):
        self.p, self.D = p, p["dim"]
        self.fluid = torch.as_tensor(np.asarray(solid) == 0, device=device)
        self.h = [p["hx"], p["hy"], p["hz"]][:self.D]
        self.V = math.prod(self.h)
        self.S = [self.V / h for h in self.h]
        kw = dict(dtype=torch.float64, device=device)
        f = self.fluid
        self.inner, self.inlet, self.outlet, self.wall_lo, self.wall_hi = [], [], [], [], []
        for a in range(self.D):
            lo, hi = self._lo(f, a), self._hi(f, a)   # the cell below / above each face, False beyond the domain
            edge_lo, edge_hi = torch.zeros_like(lo), torch.zeros_like(lo)
            edge_lo.select(self.ax(a), 0).fill_(True)
            edge_hi.select(self.ax(a), -1).fill_(True)
            self.inner.append(lo & hi)
            self.inlet.append(hi & edge_lo if a == 0 else torch.zeros_like(lo))
            self.outlet.append(lo & edge_hi if a == 0 else torch.zeros_like(lo))
            self.wall_lo.append(lo & ~hi & ~self.outlet[a])    # fluid below the face, wall above
            self.wall_hi.append(hi & ~lo & ~self.inlet[a])
        z = lambda: torch.zeros(f.shape, **kw)  # noqa: E731
        self.alpha = torch.where(f, torch.as_tensor(np.asarray(alpha0), **kw), z())
        self.zero_faces = [torch.zeros(m.shape, **kw) for m in self.inner]
        self.u = {k: [z() for _ in self.h] for k in ("vd", "cr", "sum")}
        self.q = {"vd": z(), "cr": z()}
        self.phi = {k: [x.clone() for x in self.zero_faces] for k in ("vd", "cr")}
        self.last_N = 1
        self.interface(self.alpha)

    def ax(self, a):
        return self.D - 1 - a

    def _pad(self, x, a, lo):
        s = list(x.shape)
        s[self.ax(a)] = 1
        e = torch.zeros(s, dtype=x.dtype, device=x.device)
        return torch.cat([e, x] if lo else [x, e], self.ax(a))

    def _lo(self, x, a):   # of every face, the value of the cell below it (0 beyond the domain)
        return self._pad(x, a, True)

    def _hi(self, x, a):
        return self._pad(x, a, False)

    def below(self, F, a):   # of every cell, the value of its low face
        return F.narrow(self.ax(a), 0, F.shape[self.ax(a)] - 1)

    def above(self, F, a):
        return F.narrow(self.ax(a), 1, F.shape[self.ax(a)] - 1)

    def diff(self, F, a):
        return self.above(F, a) - self.below(F, a)

    def transport(self, phi, dt):
        p, al = self.p, self.alpha
        rV = dt / self.V
        zero = torch.zeros((), dtype=al.dtype, device=al.device)
        AD, out = [], torch.zeros_like(al)
        for a in range(self.D):
            L, H, ph, inner = self._lo(al, a), self._hi(al, a), phi[a], self.inner[a]
            up = ph >= 0
            # the cell upwind of the upwind one, where the face between them is interior
            LL = self._lo(self.below(L, a), a)
            hasLL = self._lo(self.below(inner, a), a)
            HH = self._hi(self.above(H, a), a)
            hasHH = self._hi(self.above(inner, a), a)
            aU, aD = torch.where(up, L, H), torch.where(up, H, L)
            du = torch.where(torch.where(up, hasLL, hasHH), aU - torch.where(up, LL, HH), zero)
            dc = aD - aU
            mono = du * dc > 0
            vl = torch.where(mono, aU + du * dc / torch.where(mono, du + dc, 1.0), aU)
            flow = ph * aU
            phir = p["c_alpha"] * ph.abs() * self.nf[a]
            fc = torch.where(phir >= 0, phir * L * (1 - H), phir * H * (1 - L))
            AD.append(torch.where(inner, ph * vl + fc - flow, zero))
            FL = torch.where(inner, flow, zero)
            FL = torch.where(self.inlet[a], torch.where(up, ph * p["alpha_inlet"], ph * H), FL)
            FL = torch.where(self.outlet[a], ph * L, FL)
            out = out + self.diff(FL, a)
        aL = torch.where(self.fluid, al - rV * out, zero)
        hi, lo = torch.maximum(al, aL), torch.minimum(al, aL)
        inf = torch.tensor(math.inf, dtype=al.dtype, device=al.device)
        amax, amin, Pp, Pm = hi, lo, torch.zeros_like(al), torch.zeros_like(al)
        for a in range(self.D):
            inner = self.inner[a]
            for near, face in ((self._lo, self.below), (self._hi, self.above)):
                m = face(inner, a)
                amax = torch.where(m, torch.maximum(amax, face(torch.where(inner, near(hi, a), -inf), a)), amax)
                amin = torch.where(m, torch.minimum(amin, face(torch.where(inner, near(lo, a), inf), a)), amin)
            for o in (-self.below(AD[a], a), self.above(AD[a], a)):
                Pm = Pm + o.clamp(min=0)
                Pp = Pp + (-o).clamp(min=0)
        Qp = ((amax.clamp(max=1.0) - aL) / rV).clamp(min=0)
        Qm = ((aL - amin.clamp(min=0.0)) / rV).clamp(min=0)
        Rp = torch.where(Pp > 0, (Qp / torch.where(Pp > 0, Pp, 1.0)).clamp(max=1.0), zero)
        Rm = torch.where(Pm > 0, (Qm / torch.where(Pm > 0, Pm, 1.0)).clamp(max=1.0), zero)
        out = torch.zeros_like(al)
        for a in range(self.D):
            lam = torch.where(AD[a] >= 0, torch.minimum(self._lo(Rm, a), self._hi(Rp, a)),
                              torch.minimum(self._hi(Rm, a), self._lo(Rp, a)))
            out = out + self.diff(torch.where(self.inner[a], lam * AD[a], zero), a)
        return torch.where(self.fluid, aL - rV * out, zero)

    def grad(self, x, b):   # Gauss gradient, boundary faces take the cell's value
        F = torch.where(self.inner[b], 0.5 * (self._lo(x, b) + self._hi(x, b)), torch.zeros((), dtype=x.dtype, device=x.device))
        lo = torch.where(self.below(self.inner[b], b), self.below(F, b), x)
        hi = torch.where(self.above(self.inner[b], b), self.above(F, b), x)
        return (hi - lo) / self.h[b]

    def interface(self, alpha):
        p, x = self.p, alpha
        zero = torch.zeros((), dtype=x.dtype, device=x.device)
        for _ in range(p["n_smooth"]):
            num = torch.zeros_like(x)
            for a in range(self.D):
                F = 0.5 * (self._lo(x, a) + self._hi(x, a))
                for face in (self.below, self.above):
                    num = num + torch.where(face(self.inner[a], a), face(F, a), x) * self.S[a]
            x = torch.where(self.fluid, num / (2 * sum(self.S)), zero)
        delta = 1e-8 / self.V ** (1.0 / self.D)
        ct = math.cos(p["theta_deg"] * math.pi / 180.0)
        g = [self.grad(x, b) for b in range(self.D)]
        self.nf, div = [], torch.zeros_like(x)
        for a in range(self.D):
            ga = (self._hi(x, a) - self._lo(x, a)) / self.h[a]
            mag = ga * ga
            for b in range(self.D):
                if b != a:
                    mag = mag + (0.5 * (self._lo(g[b], a) + self._hi(g[b], a))) ** 2
            n = torch.where(self.inner[a], ga / (mag.sqrt() + delta), zero)
            n = torch.where(self.wall_lo[a], torch.full_like(n, ct), n)
            self.nf.append(torch.where(self.wall_hi[a], torch.full_like(n, -ct), n))
            div = div + self.diff(self.nf[a], a) / self.h[a]
        self.kappa = torch.where(self.fluid, -div, zero)

    def apply(self, cf, x):
        y = None
        for a in range(self.D):
            t = self.diff(cf[a] * (self._lo(x, a) - self._hi(x, a)), a)   # beyond the outlet x = 0; elsewhere c = 0
            y = t if y is None else y + t
        return y

    def solve(self, cf, b, q):
        m = int(self.fluid.sum())
        if m <= 3000:
            if self.dense is None:   # the operator's columns, one fluid cell at a time over batched unit fields
                idx = self.fluid.flatten().nonzero().flatten()
                A = torch.zeros((m, m), dtype=b.dtype, device=b.device)
                number = torch.full((self.fluid.numel(),), -1, dtype=torch.long, device=b.device)
                number[idx] = torch.arange(m, device=b.device)
                number = number.reshape(self.fluid.shape)
                for a in range(self.D):
                    lo, hi, c = self._lo(number, a), self._hi(number, a), cf[a]
                    k = self.inner[a]
                    i, j, w = lo[k], hi[k], c[k]
                    A.index_put_((i, j), -w, accumulate=True)
                    A.index_put_((j, i), -w, accumulate=True)
                    A.index_put_((i, i), w, accumulate=True)
                    A.index_put_((j, j), w, accumulate=True)
                    k = self.outlet[a]
                    A.index_put_((lo[k], lo[k]), c[k], accumulate=True)
                self.dense = (idx, torch.linalg.cholesky(A))
            idx, L = self.dense
            x = torch.zeros_like(b).flatten()
            x[idx] = torch.cholesky_solve(b.flatten()[idx][:, None], L)[:, 0]
            return x.reshape(b.shape)
        diag = sum(self.below(cf[a], a) + self.above(cf[a], a) for a in range(self.D))
        inv = torch.where(diag > 0, 1.0 / torch.where(diag > 0, diag, 1.0), torch.zeros_like(diag))
        q = q.clone()
        r = b - self.apply(cf, q)
        z = inv * r
        d, rz, stop = z.clone(), (r * z).sum(), (1e-14 if self.p["precision"] == FP64 else 1e-12) * b.norm()
        for it in range(20000):
            Ad = self.apply(cf, d)
            al = rz / (d * Ad).sum()
            q += al * d
            r -= al * Ad
            if it % 32 == 31 and bool(r.norm() <= stop):
                break
            z = inv * r
            new = (r * z).sum()
            d = z + (new / rz) * d
            rz = new
        return q

    def piso(self, which, alpha, phic, tension, vin0, dt):
        p, D = self.p, self.D
        v, vold, q = self.u[which], [x.clone() for x in self.u[which]], self.q[which]
        zero = torch.zeros((), dtype=alpha.dtype, device=alpha.device)
        mix = lambda x, y: torch.where(self.fluid, alpha * x + (1 - alpha) * y, zero)  # noqa: E731
        rho, mu = mix(p["rho1"], p["rho2"]), mix(p["mu1"], p["mu2"])
        acc, cin = torch.zeros_like(alpha), torch.zeros_like(alpha)
        muf = [0.5 * (self._lo(mu, a) + self._hi(mu, a)) for a in range(D)]
        for a in range(D):
            S, h = self.S[a], self.h[a]
            for face, sg in ((self.below, -1.0), (self.above, 1.0)):
                i, inl = face(self.inner[a], a), face(self.inlet[a], a)
                w = face(self.wall_lo[a] | self.wall_hi[a] | self.inlet[a], a)
                acc = acc + torch.where(i, face(muf[a], a) * S / h, torch.where(w, mu * S / (0.5 * h), zero))
                cin = cin + torch.where(i | inl, (-sg * face(phic[a], a)).clamp(min=0), zero)
        rA = torch.where(self.fluid, 1.0 / torch.where(self.fluid, rho / dt + (acc + rho * cin) / self.V, 1.0), zero)
        cf, fst = [], []
        for a in range(D):
            S, h = self.S[a], self.h[a]
            c = torch.where(self.inner[a], 0.5 * (self._lo(rA, a) + self._hi(rA, a)) * S / h, zero)
            cf.append(torch.where(self.outlet[a], self._lo(rA, a) * S / (0.5 * h), c))
            k = 0.5 * (self._lo(self.kappa, a) + self._hi(self.kappa, a))
            f = p["sigma"] * k * (self._hi(alpha, a) - self._lo(alpha, a)) / h if tension else self.zero_faces[a]
            fst.append(torch.where(self.inner[a], f, zero))
        self.dense, E = None, None
        for corr in range(p["n_piso"]):
            G = [[None] * D for _ in range(D)]
            for comp in range(D):
                x = v[comp]
                for b in range(D):
                    F = torch.where(self.inner[b], 0.5 * (self._lo(x, b) + self._hi(x, b)), zero)
                    F = torch.where(self.inlet[b], torch.full_like(F, vin0 if comp == 0 else 0.0), F)
                    F = torch.where(self.outlet[b], self._lo(x, b), F)
                    G[comp][b] = torch.where(self.fluid, self.diff(F, b) / self.h[b], zero)
            hbya = []
            for comp in range(D):
                x, vin = v[comp], vin0 if comp == 0 else 0.0
                lap, conv, tr, inflow = (torch.zeros_like(x) for _ in range(4))
                for a in range(D):
                    S, h, ph = self.S[a], self.h[a], phic[a]
                    inner, inlet = self.inner[a], self.inlet[a]
                    up = ph >= 0
                    corr_up = torch.where(up, 0.5 * h * self._lo(G[comp][a], a), -0.5 * h * self._hi(G[comp][a], a))
                    trf = torch.where(inner, muf[a] * S * 0.5 * (self._lo(G[a][comp], a) + self._hi(G[a][comp], a)), zero)
                    for face, near, sg in ((self.below, self._lo, -1.0), (self.above, self._hi, 1.0)):
                        i, inl = face(inner, a), face(inlet, a)
                        bnd = face(self.wall_lo[a] | self.wall_hi[a] | self.inlet[a] | self.outlet[a], a)
                        vn, fo = face(near(x, a), a), sg * face(ph, a)
                        lap = lap + torch.where(i, face(muf[a], a) * S / h * vn, torch.where(inl, mu * S / (0.5 * h) * vin, zero))
                        inflow = inflow + torch.where(i, (-fo).clamp(min=0) * vn, torch.where(inl, (-fo).clamp(min=0) * vin, zero))
                        conv = conv + torch.where(i, fo * face(corr_up, a), torch.where(inl & (fo >= 0), fo * (vin - x), zero))
                        tr = tr + torch.where(i, sg * face(trf, a), torch.where(bnd, sg * mu * S * G[a][comp], zero))
                H = rho * vold[comp] / dt + (lap + rho * (inflow - conv) + tr) / self.V
                hbya.append(rA * H)
            phis, b = [], torch.zeros_like(alpha)
            for a in range(D):
                S = self.S[a]
                F = torch.where(self.inner[a], 0.5 * (self._lo(hbya[a], a) + self._hi(hbya[a], a)) * S
                                + 0.5 * (self._lo(rA, a) + self._hi(rA, a)) * fst[a] * S, zero)
                F = torch.where(self.inlet[a], torch.full_like(F, (vin0 if a == 0 else 0.0) * S), F)
                phis.append(torch.where(self.outlet[a], self._lo(hbya[a], a) * S, F))
                b = b - self.diff(phis[a], a)
            b = torch.where(self.fluid, b, zero)
            if corr == 0:   # the normalised initial residual of the exit test
                Mq = self.apply(cf, q)
                Mbar = torch.where(self.fluid, self.apply(cf, torch.where(self.fluid, q.sum() / self.fluid.sum(), zero)), zero)
                E = float((b - Mq).abs().sum() / ((Mq - Mbar).abs().sum() + (b - Mbar).abs().sum() + 1e-20))
            q = self.solve(cf, b, q)
            phi = [phis[a] - cf[a] * (self._hi(q, a) - self._lo(q, a)) for a in range(D)]
            v = []
            for a in range(D):
                F = fst[a] - (self._hi(q, a) - self._lo(q, a)) / self.h[a]
                F = torch.where(self.inner[a], F, torch.where(self.outlet[a], self._lo(q, a) / (0.5 * self.h[a]), zero))
                v.append(hbya[a] + rA * 0.5 * (self.below(F, a) + self.above(F, a)))
        self.u[which], self.q[which], self.phi[which] = v, q, phi
        return E, vold

    def drag(self, dt):
        new = self.transport(self.phi["vd"], dt)
        phic = [x + y for x, y in zip(self.phi["vd"], self.phi["cr"])]
        self.piso("vd", new, phic, False, self.p["U_inlet"], dt)
        self.alpha = new
        self.interface(new)

    def standard(self, dt):
        new = self.transport(self.phi["vd"], dt)
        self.interface(new)
        self.piso("vd", new, self.phi["vd"], True, self.p["U_inlet"], dt)
        self.alpha = new

    def relax(self, dt, N):
        self.u["sum"], self.last_N = [torch.zeros_like(self.alpha) for _ in self.h], N
        for _ in range(N):
            new = self.transport(self.phi["cr"], dt)
            self.interface(new)
            phic = [x + y for x, y in zip(self.phi["vd"], self.phi["cr"])]
            E, old = self.piso("cr", new, phic, True, 0.0, dt)
            self.alpha = new
            self.u["sum"] = [s + x for s, x in zip(self.u["sum"], self.u["cr"])]
            if self.p["conv_mode"] == inputs.CONV_DU_MAX:
                E = float(max((x - y).abs().max() for x, y in zip(self.u["cr"], old))) / self.p["U_inlet"]
            if E < self.p["conv_tol"]:
                break

    def snapshot(self, step):
        d = {"alpha": self.alpha, "p": self.q["vd"] + self.q["cr"]}
        for a in range(self.D):
            d["u" + "xyz"[a]] = self.u["vd"][a] + self.u["sum"][a] / self.last_N
            d["phi" + "xyz"[a]] = self.phi["vd" if step == "standard" else "cr"][a]
        return d


def exact(case, seed):
    # seconds, from the growth of the iterations with the extent along x and of an iteration with the cells
    cells = case["nx"] * case["ny"] * case["nz"]
    one = (1.8 if case["nz"] > 1 else 2.9 * case["nx"] / 1024) * max(1.0, cells / 1.5e6)
    if cells > 3000 and (1 + case["sub"]) * one * (0.5 * case["inst"] if case["step"] == "batch" else 1) > 20:
        return None
    device = "cuda" if torch.cuda.is_available() else "cpu"
    got = []
    for q in range(case["inst"]):
        c = _make(case, seed, q)
        dt_vd, dt_cr = _steps(c.params, case["sub"])
        s = _Exact(c.params, c.solid, c.alpha0, device)
        if case["step"] == "standard":
            s.standard(dt_cr)
        else:
            s.drag(dt_vd)
            s.relax(dt_cr, case["sub"])
        got.append(s.snapshot(case["step"]))
    return got if case["step"] == "batch" else got[0]

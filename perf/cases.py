"""The solves whose speed is followed, as a program that uses the library makes
them: a problem and its host FP64 initial fields, one ``hydro.Simulation`` or
``hydro.Batch`` with the library's default configuration, and a few time steps
per pass.

* ``listed()``  the followed cases: the smallest calls (launch latency), the
  ordinary ones and the largest, 2D and 3D, FP64 and FP32, every integrator and
  reconstruction, the hydrostatic background, ragged grids, a mixed batch and a
  whole solve from host arrays to host arrays.
* ``draw(rng)``  one more case of the same ranges.
* ``prepare(case, seed)``  the problem, seeded fields and the handle.
* ``run(state)``  one pass; returns the whole state it reached.
* ``work(case)``  bytes and floating-point operations the pass cannot do without.
* ``exact(case, seed)``  the same pass in FP64 with plain torch operations: the
  scheme's textbook formulas on whole padded arrays.

A pass continues from the state the previous one reached, as a time loop does.
"""

from __future__ import annotations

import math

import numpy as np
import torch

from paper_1510_05061_gb300 import hydro, inputs

SCHEMES = {"hancock": inputs.HANCOCK, "rk2": inputs.SSPRK2, "ctu": inputs.CTU}
RECONS = {"plm": inputs.PLM, "ppm": inputs.PPM}
# scheme operations per zone and step, each face once (divisions, square
# roots, minima and maxima count as one): (2D, 3D)
FLOPS = {("hancock", "plm"): (321, 542), ("rk2", "plm"): (531, 903), ("rk2", "ppm"): (771, 1353),
         ("ctu", "plm"): (553, 1032)}


def _case(name, kind="steps", family="rt", nx=64, ny=64, nz=64, precision="fp64", hse=0, scheme="hancock",
          recon="plm", steps=2, boxes=0):
    c = dict(kind=kind, family=family, nx=nx, ny=ny, nz=nz, precision=precision, hse=hse, scheme=scheme,
             recon=recon, steps=steps, boxes=boxes)
    return c if name is None else dict(c, name=name)


def listed():
    return [
        # the smallest call: one step of the standard 128^2 shock tube, enqueued by itself
        _case("sod2d_128_fp64", family="sod", nx=128, ny=128, nz=1, steps=1),
        # a small 3D box of a parameter study, launch-bound
        _case("kh3d_32_fp32", family="kh", nx=32, ny=32, nz=32, precision="fp32", steps=2),
        # an ordinary 2D run in FP64, odd extents
        _case("kh2d_517x331_fp64", family="kh", nx=517, ny=331, nz=1, steps=2),
        # a large 2D run in FP32
        _case("kh2d_2048_fp32", family="kh", nx=2048, ny=2048, nz=1, precision="fp32", steps=2),
        # a small stratified run driven by advance_to, with the conserved totals
        # after each batch of steps (the host waits)
        _case("rt3d_64_fp64_hse_diag", kind="advance", nx=64, ny=64, nz=64, hse=1, steps=4),
        # the benchmark's Rayleigh-Taylor box
        _case("rt3d_256_fp64", nx=256, ny=256, nz=256, steps=1),
        # the largest: the FP32 precision mode on perturbations of the background
        _case("rt3d_320_fp32_hse", nx=320, ny=320, nz=320, precision="fp32", hse=1, steps=2),
        # a walled box under oblique gravity, ragged against every tile
        _case("walls3d_101x75x130_fp64", family="walls", nx=101, ny=75, nz=130, steps=2),
        # the accurate integrators: piecewise parabolic method of lines, corner transport upwind
        _case("rt3d_128_fp64_rk2_ppm", nx=128, ny=128, nz=128, scheme="rk2", recon="ppm", steps=1),
        _case("rt3d_128_fp64_ctu", nx=128, ny=128, nz=128, scheme="ctu", steps=1),
        # a capacity run: uneven 3D and 2D boxes stepping together
        _case("kh_batch_fp32", kind="batch", family="kh", nx=32, ny=128, nz=0, precision="fp32", steps=4, boxes=14),
        # a whole solve, host arrays in and out
        _case("rt3d_96_fp32_hse_solve", kind="solve", nx=96, ny=96, nz=96, precision="fp32", hse=1, steps=20),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choices(["steps", "advance", "batch", "solve"], [8, 1, 2, 1])[0]
    precision = rng.choice(["fp64", "fp32"])
    if kind == "batch":
        lo = _log_int(rng, 16, 40)
        return _case(None, kind="batch", family="kh", nx=lo, ny=_log_int(rng, 64, 144), nz=0, precision="fp32",
                     steps=2 * rng.randint(1, 3), boxes=rng.randint(4, 16))
    dim3 = rng.random() < 0.7
    scheme, recon = rng.choices([("hancock", "plm"), ("rk2", "plm"), ("rk2", "ppm"), ("ctu", "plm")], [5, 1, 1, 1])[0]
    # zone-steps of one pass: no more than the largest listed case's time
    cap = (12e6 if precision == "fp64" else 40e6) * 542 / FLOPS[scheme, recon][1]
    if dim3:
        family = rng.choice(["rt", "kh", "walls"])
        hi = 240 if precision == "fp64" else 320
        nx, ny, nz = (_log_int(rng, 16, hi) for _ in range(3))
        hse = 0
        if family == "rt":
            ny = nx
            hse = int(recon == "plm" and rng.random() < 0.6)
    else:
        family, nz, hse = rng.choice(["sod", "kh", "walls"]), 1, 0
        nx, ny = (_log_int(rng, 48, 2600) for _ in range(2))
    steps = rng.randint(1, 4)
    while nx * ny * nz * steps > cap:
        if steps > 1:
            steps -= 1
        elif dim3:
            nz = nz * 3 // 4
        else:
            ny = ny * 3 // 4
    if kind == "solve" and nx * ny * nz > 1e6:
        kind = "steps"
    return _case(None, kind=kind, family=family, nx=nx, ny=ny, nz=nz, precision=precision, hse=hse, scheme=scheme,
                 recon=recon, steps=steps)


# ------------------------------------------------------------------ inputs

def _walls(nx, ny, nz, seed):
    """A closed box (reflecting walls) under oblique gravity: smooth density
    and velocity modes, seeded amplitudes and phases."""
    ndim = 3 if nz > 1 else 2
    ns = (nx, ny, nz)
    wall = (inputs.BC_REFLECT,) * 3
    prob = inputs.Problem(ndim=ndim, n=ns, hi=(1.0, 0.75, 1.25 if ndim == 3 else 1.0), bc_lo=wall, bc_hi=wall,
                          grav=(0.2, -0.3, -0.5 if ndim == 3 else 0.0), name=f"walls-{nx}x{ny}x{nz}")
    u = inputs.draw_uniform(seed, 41, np.arange(64)).reshape(8, 8)
    axes = [2.0 * math.pi * (prob.centres(d) - prob.lo[d]) / (prob.hi[d] - prob.lo[d]) for d in range(ndim)]
    W = np.zeros(prob.shape)
    for q in range(ndim + 2):
        f = np.zeros(prob.shape[1:])
        for d in range(ndim):
            s = [1, 1, 1]
            s[2 - d] = -1
            f = f + (u[q, d] * np.cos((1 + (q + d) % 3) * axes[d] + 6.0 * u[q, 3 + d])).reshape(s)
        W[q] = 0.1 * f
    W[0] += 1.0
    W[-1] += 2.5
    return prob, W


def _shear(nx, ny, nz, precision, seed):
    """The periodic double shear layer on an nx x ny x nz grid: seeded jump,
    density ratio and per-cell noise."""
    u = inputs.draw_uniform(seed, 42, np.arange(2))
    per = (inputs.BC_PERIODIC,) * 3
    prob = inputs.Problem(ndim=3 if nz > 1 else 2, n=(nx, ny, nz), bc_lo=per, bc_hi=per, precision=precision,
                          name=f"kh-{nx}x{ny}x{nz}")
    y = prob.centres(1)
    prof = 0.5 * (np.tanh((y - 0.25) / 0.025) - np.tanh((y - 0.75) / 0.025))
    W = np.zeros(prob.shape)
    W[0] = (1.0 + (1.0 + float(u[0])) * prof)[None, :, None]
    W[1] = ((0.75 + float(u[1])) * (prof - 0.5))[None, :, None]
    W[2] = 0.01 * (2.0 * np.random.default_rng(seed).random(prob.shape[1:]) - 1.0)
    W[-1] = 2.5
    return prob, W


def _problem(case, seed):
    """The problem and host FP64 primitives of a single-solve case."""
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    prec = inputs.FP32 if case["precision"] == "fp32" else inputs.FP64
    if case["family"] == "rt":
        prob, W = inputs.rayleigh_taylor(nx, seed=seed, nz=nz, hse_subtract=case["hse"])
    elif case["family"] == "kh":
        prob, W = _shear(nx, ny, nz, prec, seed)
    elif case["family"] == "walls":
        prob, W = _walls(nx, ny, nz, seed)
    else:
        prob, W = inputs.sod(4)
        u = inputs.draw_uniform(seed, 43, np.arange(2))
        prob = prob.replace(n=(nx, ny, nz), name=f"sod2d-{nx}x{ny}")
        left = (prob.centres(0) < 0.5)[None, None, :]
        W = np.zeros(prob.shape)
        W[0] = np.where(left, 0.9 + 0.2 * u[0], 0.125)
        W[-1] = np.where(left, 0.9 + 0.2 * u[1], 0.1)
    return prob.replace(precision=prec, scheme=SCHEMES[case["scheme"]], recon=RECONS[case["recon"]]), W


def _boxes(case):
    """(nx, ny, nz) of a batch's boxes: 3D cubes log-spaced over the case's
    range, every fourth box a 2D grid."""
    n, lo, hi = case["boxes"], case["nx"], case["ny"]
    out = []
    for i in range(n):
        s = int(round(lo * (hi / lo) ** (i / max(n - 1, 1))))
        out.append((s, s, s) if i % 4 != 3 else (4 * s + i, 3 * s, 1))
    return out


def _batch_items(case, seed):
    return [_shear(nx, ny, nz, inputs.FP32, seed + 1000 * i) for i, (nx, ny, nz) in enumerate(_boxes(case))]


class _Buffer:
    """A state buffer as the CUDA array interface describes it; a tensor made
    from it keeps the handle that owns the memory."""

    def __init__(self, owner, ptr, prob):
        self.owner = owner
        self.__cuda_array_interface__ = {"shape": prob.shape, "version": 3, "data": (ptr, False),
                                         "typestr": "<f4" if prob.precision == inputs.FP32 else "<f8"}


def _current(state):
    """The solve's current state as a tensor (one per ping-pong buffer)."""
    sim, views = state["sim"], state["views"]
    ptr = sim.current_ptr()
    if ptr not in views:
        views[ptr] = torch.as_tensor(_Buffer(sim, ptr, sim.prob), device="cuda")
    return views[ptr]


# -------------------------------------------------------------------- cases

def prepare(case, seed):
    if case["kind"] == "batch":
        batch = hydro.Batch(_batch_items(case, seed))
        # an even number of steps leaves each instance's state in the buffer it starts from
        outs = [torch.as_tensor(_Buffer(batch, hydro.load().hydro_batch_current(batch.h, i), p), device="cuda")
                for i, p in enumerate(batch.probs)]
        return {"case": case, "batch": batch, "outs": outs}
    prob, W = _problem(case, seed)
    if case["kind"] == "solve":
        return {"case": case, "prob": prob, "W": W}
    return {"case": case, "sim": hydro.Simulation(prob, W), "views": {}}


def run(state):
    case = state["case"]
    if case["kind"] == "batch":
        state["batch"].step(case["steps"])
        return state["outs"]
    if case["kind"] == "solve":
        sim = hydro.Simulation(state["prob"], state["W"])
        sim.run_steps(case["steps"])
        out = {"U": sim.conserved(), "totals": sim.totals()}
        sim.close()
        return out
    sim = state["sim"]
    if case["kind"] == "advance":
        _, t = sim.advance_to(1e6, max_steps=case["steps"])
        totals = sim.totals()
        return {"U": _current(state), "t": t, "totals": totals}
    sim.run_steps(case["steps"])
    return _current(state)


def work(case):
    size = 4 if case["precision"] == "fp32" else 8
    grids = _boxes(case) if case["kind"] == "batch" else [(case["nx"], case["ny"], case["nz"])]
    nbytes = flops = 0.0
    for nx, ny, nz in grids:
        d3 = nz > 1
        zones, nv = nx * ny * nz, 5 if d3 else 4
        # one read and one write of the state per step; the method of lines
        # reads U^n and writes U1, then reads both and writes U^{n+1}
        passes = 5 if case["scheme"] == "rk2" else 2
        nbytes += case["steps"] * passes * nv * size * zones
        flops += case["steps"] * FLOPS[case["scheme"], case["recon"]][d3] * zones
        if case["kind"] == "solve":
            nbytes += 16 * nv * zones
    return {"bytes": nbytes, "flops": flops}


# ------------------------------------------------- the scheme in plain torch

class _Reference:
    """The update of one problem on whole arrays (nvar, nz, ny, nx), FP64."""

    def __init__(self, prob):
        self.p, self.nd, self.nv = prob, prob.ndim, prob.ndim + 2
        self.n, self.dx, self.dev = prob.n, prob.dx(), "cuda" if torch.cuda.is_available() else "cpu"
        self.ng = 3 if prob.recon == inputs.PPM else 2
        self.hse = bool(prob.hse_subtract)
        zero = torch.zeros(1, dtype=torch.float64, device=self.dev)

        def table(a):
            return torch.as_tensor(np.asarray(a), device=self.dev).view(-1, 1, 1) if self.hse else zero

        self.rc, self.pc, self.rf, self.pf = (table(a) for a in (prob.bg_rho_c, prob.bg_p_c, prob.bg_rho_f,
                                                                 prob.bg_p_f))
        # background of the ring planes -1 .. nz: centre, low and high face
        if self.hse:
            nz = prob.n[2]
            self.ring = dict(rho=self.rc[1:nz + 3], p=self.pc[1:nz + 3], rlo=self.rf[1:nz + 3],
                             rhi=self.rf[2:nz + 4], plo=self.pf[1:nz + 3], phi=self.pf[2:nz + 4])
        else:
            self.ring = dict.fromkeys(("rho", "p", "rlo", "rhi", "plo", "phi"), zero)
        r = self.ring
        self.B = (r["phi"] - r["plo"]) / self.dx[2] - r["rho"] * prob.grav[2] if self.hse else zero

    def inner_planes(self, a):
        return a[1:-1] if self.hse else a

    # conserved and primitive variables
    def to_cons(self, W):
        ke = (W[1:-1] ** 2).sum(0)
        U = torch.empty_like(W)
        U[0], U[1:-1] = W[0], W[0] * W[1:-1]
        U[-1] = W[-1] / (self.p.gamma - 1.0) + 0.5 * W[0] * ke
        if self.hse:
            U[0] -= self.rc[2:-2]
            U[-1] -= self.pc[2:-2] / (self.p.gamma - 1.0)
        return U

    def to_prim(self, U, rho_bg):
        W = torch.empty_like(U)
        rho = rho_bg + U[0]
        W[0], W[1:-1] = U[0], U[1:-1] / rho
        W[-1] = (self.p.gamma - 1.0) * (U[-1] - 0.5 * (U[1:-1] ** 2).sum(0) / rho)
        return W

    def dt(self, U):
        W = self.to_prim(U, self.rc[2:-2] if self.hse else 0.0)
        rho = W[0] + (self.rc[2:-2] if self.hse else 0.0)
        pr = W[-1] + (self.pc[2:-2] if self.hse else 0.0)
        c = torch.sqrt(self.p.gamma * pr / rho)
        s = sum((W[1 + d].abs() + c) / self.dx[d] for d in range(self.nd))
        return self.p.cfl / float(s.max())

    # ghost cells and shifted views
    def pad(self, W):
        for d in range(self.nd):
            n, lo, hi = self.n[d], self.p.bc_lo[d], self.p.bc_hi[d]
            idx, sgn = [], []
            for g in range(-self.ng, n + self.ng):
                bc = lo if g < 0 else hi if g >= n else None
                m, s = g, 1.0
                if bc == inputs.BC_PERIODIC:
                    m = g % n
                elif bc == inputs.BC_REFLECT:
                    m, s = (-1 - g if g < 0 else 2 * n - 1 - g), -1.0
                elif bc is not None:
                    m = 0 if g < 0 else n - 1
                idx.append(m)
                sgn.append(s)
            W = W.index_select(3 - d, torch.tensor(idx, device=self.dev))
            shape = [1, 1, 1]
            shape[2 - d] = -1
            W[1 + d] *= torch.tensor(sgn, dtype=torch.float64, device=self.dev).view(shape)
        return W

    def at(self, Wp, d=0, s=0):
        """The cells -1 .. n of every active axis, shifted by s along d."""
        for e in range(self.nd):
            Wp = Wp.narrow(3 - e, self.ng - 1 + (s if e == d else 0), self.n[e] + 2)
        return Wp

    @staticmethod
    def mc(dl, dr):
        a = torch.minimum(2.0 * torch.minimum(dl.abs(), dr.abs()), 0.5 * (dl + dr).abs())
        return torch.where((dl.sign() * dr.sign()) > 0, torch.copysign(a, dr), torch.zeros_like(a))

    def slope(self, Wp, d, s=0):
        w = self.at(Wp, d, s)
        return self.mc(w - self.at(Wp, d, s - 1), self.at(Wp, d, s + 1) - w)

    # face states [(low, high)] per axis on the ring cells
    def faces(self, Wp, dt, mode):
        p, nd, b = self.p, self.nd, self.ring
        w = self.at(Wp)
        rho, pr, gam, hdt = b["rho"] + w[0], b["p"] + w[-1], p.gamma, 0.5 * dt
        if p.recon == inputs.PPM:
            out = []
            for d in range(nd):
                sm, s0, sp = (self.slope(Wp, d, k) for k in (-1, 0, 1))
                am, ap = self.at(Wp, d, -1), self.at(Wp, d, 1)
                lo, hi = 0.5 * (am + w) - (s0 - sm) / 6.0, 0.5 * (w + ap) - (sp - s0) / 6.0
                flat = (hi - w) * (w - lo) <= 0.0
                da, a6 = hi - lo, 6.0 * (w - 0.5 * (lo + hi))
                fl = ~flat & (da * a6 > da * da)
                fr = ~flat & ~fl & (-(da * da) > da * a6)
                out.append((torch.where(flat, w, torch.where(fl, 3.0 * w - 2.0 * hi, lo)),
                            torch.where(flat, w, torch.where(fr, 3.0 * w - 2.0 * lo, hi))))
            return out
        dw = [self.slope(Wp, d) for d in range(nd)]

        def along(d):
            un, r = w[1 + d], torch.zeros_like(w)
            r[0] = -(un * dw[d][0] + rho * dw[d][1 + d]) / self.dx[d]
            for e in range(nd):
                r[1 + e] = -un * dw[d][1 + e] / self.dx[d]
            r[1 + d] -= dw[d][-1] / rho / self.dx[d]
            r[-1] = -(un * dw[d][-1] + gam * pr * dw[d][1 + d]) / self.dx[d]
            if self.hse and d == 2:
                r[0] -= w[3] * (b["rhi"] - b["rlo"]) / self.dx[2]
                r[-1] -= w[3] * (b["phi"] - b["plo"]) / self.dx[2]
            return r

        # source of the half step on the velocities: g rho'/rho (- B/rho), or plain g
        src, plain = torch.zeros_like(w), torch.zeros_like(w)
        for e in range(nd):
            src[1 + e] = p.grav[e] * (w[0] / rho) if self.hse else p.grav[e]
            plain[1 + e] = p.grav[e]
        if self.hse:
            src[3] -= self.B / rho
        if mode == "stage":
            cen = [w] * nd
        elif mode == "ctu":
            cen = [w + hdt * (along(d) + (src if d == 2 else plain)) for d in range(nd)]
        else:
            wh = w + hdt * (sum(along(d) for d in range(nd)) + src)
            cen = [wh] * nd
        out, ok = [], torch.ones_like(rho, dtype=torch.bool)
        for d in range(nd):
            lo, hi = cen[d] - 0.5 * dw[d], cen[d] + 0.5 * dw[d]
            for f, r, q in ((lo, "rlo", "plo"), (hi, "rhi", "phi")):
                rb, pb = (b[r], b[q]) if d == 2 else (b["rho"], b["p"])
                ok &= (rb + f[0] > 0.0) & (pb + f[-1] > 0.0)
            out.append((lo, hi))
        if not bool(ok.all()):
            for d in range(nd):
                w0 = w
                if mode != "stage":
                    w0 = w + hdt * (plain if mode == "ctu" and d < 2 else src)
                out[d] = tuple(torch.where(ok, f, w0) for f in out[d])
        return out

    def hllc(self, wl, wr, d, rb, pb):
        gam, nd = self.p.gamma, self.nd
        side = []
        for w in (wl, wr):
            r, q = rb + w[0], pb + w[-1]
            side.append((r, q, w[1 + d], torch.sqrt(gam * q / r)))
        (rl, pl, ul, cl), (rr, pr, ur, cr) = side
        sl, sr = torch.minimum(ul - cl, ur - cr), torch.maximum(ul + cl, ur + cr)
        ml, mr = rl * (sl - ul), rr * (sr - ur)
        ss = (wr[-1] - wl[-1] + ml * ul - mr * ur) / (ml - mr)
        left = (sl >= 0) | ((sr > 0) & (ss >= 0))
        star = (sl < 0) & (sr > 0)
        w = torch.where(left, wl, wr)
        r, q = torch.where(left, rl, rr), torch.where(left, pl, pr)
        s, u = torch.where(left, sl, sr), w[1 + d]
        e = q / (gam - 1.0) + 0.5 * r * sum(w[1 + k] ** 2 for k in range(nd))
        f = torch.empty_like(w)
        f[0] = r * u
        for k in range(nd):
            f[1 + k] = r * u * w[1 + k]
        f[1 + d] += w[-1]
        f[-1] = u * (e + q)
        # F* = F + S (U* - U)
        rs = r * (s - u) / (s - ss)
        f[0] += torch.where(star, s * (rs - r), 0.0)
        for k in range(nd):
            vs = ss if k == d else w[1 + k]
            f[1 + k] += torch.where(star, s * (rs * vs - r * w[1 + k]), 0.0)
        es = rs * (e / r + (ss - u) * (ss + q / (r * (s - u))))
        f[-1] += torch.where(star, s * (es - e), 0.0)
        return f

    def flux(self, faces, d, ring):
        """Fluxes through the n + 1 faces along d, on the interior rows of
        the other axes or (ring) one row wider."""
        n, dim = self.n[d], 3 - d
        wl, wr = faces[d][1].narrow(dim, 0, n + 1), faces[d][0].narrow(dim, 1, n + 1)
        for e in range(self.nd):
            if e != d and not ring:
                wl, wr = wl.narrow(3 - e, 1, self.n[e]), wr.narrow(3 - e, 1, self.n[e])
        if self.p.bc_lo[d] == inputs.BC_REFLECT:
            wl = wl.clone()
            m = wr.select(dim, 0).clone()
            m[1 + d] *= -1.0
            wl.select(dim, 0).copy_(m)
        if self.p.bc_hi[d] == inputs.BC_REFLECT:
            wr = wr.clone()
            m = wl.select(dim, n).clone()
            m[1 + d] *= -1.0
            wr.select(dim, n).copy_(m)
        rb = pb = 0.0
        if self.hse:
            nz = self.n[2]
            if d == 2:
                rb, pb = self.rf[2:nz + 3], self.pf[2:nz + 3]
            else:
                rb, pb = (self.rc[1:-1], self.pc[1:-1]) if ring else (self.rc[2:-2], self.pc[2:-2])
        return self.hllc(wl, wr, d, rb, pb)

    def correct(self, faces, dt):
        """Transverse corrections of the one-dimensional states (ring cells
        along d, interior rows across)."""
        p, b = self.p, self.ring
        first = [self.flux(faces, d, True) for d in range(self.nd)]
        diff = [f.narrow(3 - d, 1, self.n[d]) - f.narrow(3 - d, 0, self.n[d]) for d, f in enumerate(first)]
        out = []
        for d in range(self.nd):
            pair, ok = [], True

            def rows(a, shift=0):   # interior rows of the axes other than d
                for e in range(self.nd):
                    if e != d and a.shape[3 - shift - e] == self.n[e] + 2:
                        a = a.narrow(3 - shift - e, 1, self.n[e])
                return a

            for s in (0, 1):
                w = rows(faces[d][s])
                rb, pb = (b[("rlo", "rhi")[s]], b[("plo", "phi")[s]]) if d == 2 else (b["rho"], b["p"])
                if self.hse:
                    rb, pb = rows(rb, 1), rows(pb, 1)
                r = rb + w[0]
                U = torch.empty_like(w)
                U[0], U[1:-1] = w[0], r * w[1:-1]
                U[-1] = w[-1] / (p.gamma - 1.0) + 0.5 * r * (w[1:-1] ** 2).sum(0)
                for e in range(self.nd):
                    if e == d:
                        continue
                    k = 0.5 * dt / self.dx[e]
                    U -= k * rows(diff[e])
                    if self.hse and e == 2:
                        U[3] -= k * rows(b["phi"] - b["plo"], 1)
                v = self.to_prim(U, rb)
                ok = (rb + v[0] > 0.0) & (pb + v[-1] > 0.0) & ok
                pair.append((w, v))
            new = []
            for w, v in pair:
                full = torch.where(ok, v, w)
                for e in range(self.nd):   # back to the ring layout
                    if e != d:
                        pads = [0] * 6
                        pads[2 * e:2 * e + 2] = 1, 1
                        full = torch.nn.functional.pad(full, pads)
                new.append(full)
            out.append(tuple(new))
        return out

    def update(self, U, dt, mode):
        p, nd = self.p, self.nd
        W = self.pad(self.to_prim(U, self.rc[2:-2] if self.hse else 0.0))
        faces = self.faces(W, dt, mode)
        if mode == "ctu":
            faces = self.correct(faces, dt)
        du, msrc = torch.zeros_like(U), 0.0
        for d in range(nd):
            f = self.flux(faces, d, False)
            lo, hi = f.narrow(3 - d, 0, self.n[d]), f.narrow(3 - d, 1, self.n[d])
            du -= (hi - lo) / self.dx[d]
            msrc = msrc + p.grav[d] * 0.5 * (lo[0] + hi[0])
        new = U + dt * du
        r = U[0] if mode == "stage" else 0.5 * (U[0] + new[0])
        for d in range(nd):
            new[1 + d] += dt * p.grav[d] * r
        if self.hse:
            new[3] -= dt * self.inner_planes(self.B)
        new[-1] += dt * msrc
        return new

    def step(self, U):
        dt = self.dt(U)
        if self.p.scheme == inputs.SSPRK2:
            U1 = self.update(U, dt, "stage")
            return 0.5 * (U + self.update(U1, dt, "stage")), dt
        return self.update(U, dt, "ctu" if self.p.scheme == inputs.CTU else "hancock"), dt

    def run(self, W0, steps):
        U, t = self.to_cons(torch.as_tensor(W0, device=self.dev)), 0.0
        for _ in range(steps):
            U, dt = self.step(U)
            t += dt
        return U, t

    def total(self, U):
        V = U.clone()
        if self.hse:
            V[0] += self.rc[2:-2]
            V[-1] += self.pc[2:-2] / (self.p.gamma - 1.0)
        return V

    def totals(self, U):
        vol = math.prod(self.dx[:self.nd])
        return self.total(U).sum((1, 2, 3)) * vol


def exact(case, seed):
    if case["kind"] == "batch":
        return [_Reference(p).run(W, case["steps"])[0] for p, W in _batch_items(case, seed)]
    prob, W = _problem(case, seed)
    ref = _Reference(prob)
    U, t = ref.run(W, case["steps"])
    if case["kind"] == "solve":
        return {"U": ref.total(U).cpu().numpy(), "totals": ref.totals(U).cpu().numpy()}
    if case["kind"] == "advance":
        return {"U": U, "t": t, "totals": ref.totals(U).cpu().numpy()}
    return U

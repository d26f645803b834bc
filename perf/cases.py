"""Performance cases of the LBFS solver, each one pass through lbfs.Solver.

A case is a dict of plain values; its "kind" says what a pass does:

  march    a freezing run between two outputs: `calls` calls of step(`steps`), each
           returning its statistics, then the evolved state read into host memory
  batch    the same for the first `ncase` cases of the seeded sweep, advanced together
  restart  a run resumed from a checkpoint: the state uploaded, step(`steps`), and the
           evolved state read back
  monitor  the Sec. 5 diagnostics and the derived fields of a stored state
  pseudo   `steps` pseudo-time steps of the paper's own magnetic solver

States are half-way through a freezing run: a sessile drop whose interface is slightly
deformed, frozen up to an uneven front, with a moving liquid and an uneven pressure.
A program in mixed precision keeps its outputs in 32 bits, one in FP64 in 64.
"""
import math
import random

import numpy as np
import torch

from paper_2511_10257_gb300 import inputs as I
from paper_2511_10257_gb300 import lbfs

STATE = sorted([I.PHI, I.HE, I.P, I.C, I.MX, I.MY])
CHECKPOINT = sorted(STATE + [I.FSPREV])
DERIVED = sorted([I.T, I.FL, I.U, I.V, I.MUC, I.RHO])
STATS = ("sum_C", "sum_He", "sum_Fl_drop", "n_drop", "Q_L", "t")


def _case(kind, precision, nx, ny, **kw):
    d = dict(kind=kind, precision=precision, nx=nx, ny=ny, calls=1, steps=1, graph=True, autotune=False,
             radius=0.375 * ny, angle=90.0, bo=1.0, ste=0.1, chi=1.0, theta=90.0, dts=0.5, periodic_x=False,
             mag_bc=0, gravity=0.0, ncase=1)
    d.update(kw)
    return d


def listed():
    return [
        # interactive use and coupling to another program: one step a call, its statistics looked at each time
        dict(_case("march", "mixed", 128, 64, calls=10, bo=0.5), name="small_step_by_step"),
        # a parameter study on the smallest grid, and its reference in full precision
        dict(_case("march", "mixed", 128, 64, steps=50, bo=0.5), name="small_mixed"),
        dict(_case("march", "fp64", 128, 64, steps=20, bo=0.5), name="small_fp64"),
        # the usual production grids, with output every few dozen steps
        dict(_case("march", "mixed", 512, 256, steps=50), name="medium_mixed"),
        dict(_case("march", "fp64", 512, 256, steps=10), name="medium_fp64"),
        dict(_case("march", "mixed", 1024, 512, steps=30, angle=0.0, bo=1.5, ste=0.05, chi=2.0), name="large_mixed"),
        # a wetting study: sizes that fit no tile, a contact angle, gravity, a streaming step off one half,
        # steps launched without a graph
        dict(_case("march", "mixed", 505, 253, steps=30, angle=35.0, bo=1.2, ste=0.15, theta=64.0, dts=0.4,
                   gravity=-1e-5, graph=False), name="ragged_wetting_mixed"),
        # the largest grid, tuned as the benchmark does it, and its reference in full precision
        dict(_case("march", "mixed", 4096, 2048, steps=30, angle=45.0, autotune=True), name="huge_mixed"),
        dict(_case("march", "fp64", 4096, 2048, steps=2, angle=45.0), name="huge_fp64"),
        # the seeded sweep as one batch, tuned as the benchmark does it
        dict(_case("batch", "mixed", 512, 256, steps=20, autotune=True, ncase=64), name="sweep_mixed"),
        # resuming from a checkpoint
        dict(_case("restart", "mixed", 1024, 512, steps=10, angle=0.0, bo=1.5, ste=0.05, chi=2.0), name="restart_mixed"),
        # diagnostics and derived fields between two stretches of a run
        dict(_case("monitor", "mixed", 1024, 512, angle=0.0, bo=1.5, ste=0.05, chi=2.0), name="monitor_mixed"),
    ]


def draw(rng):
    kind = rng.choice(["march"] * 7 + ["batch", "restart", "monitor", "pseudo"])
    precision = rng.choice(["mixed", "mixed", "fp64"])
    phys = dict(angle=rng.uniform(0.0, 90.0), bo=rng.uniform(0.2, 2.0), ste=rng.uniform(0.05, 0.2),
                chi=rng.choice([1.0, 1.0, 2.0]), theta=rng.choice([90.0, 90.0, 64.0, 98.0]),
                dts=rng.choice([0.5, 0.5, 0.5, 0.4]), gravity=rng.choice([0.0, -1e-5]), graph=rng.random() < 0.8)
    if kind == "pseudo":
        nx = round(math.exp(rng.uniform(math.log(64), math.log(512))))
        return _case(kind, precision, nx, nx // 2, steps=rng.randint(200, 1000), **phys)
    if kind == "batch":
        ncase = rng.randint(4, 64)
        steps = rng.randint(5, 20) if precision == "mixed" else 1
        return _case(kind, precision, 512, 256, steps=steps, ncase=ncase, autotune=rng.random() < 0.5)
    # cells times steps stay within the largest listed cases
    top = 4096 * 2048 * (30 if precision == "mixed" else 2)
    nx = round(math.exp(rng.uniform(math.log(64), math.log(4096))))
    ny = max(16, min(2048, round(nx * rng.uniform(0.3, 0.7))))
    periodic = rng.random() < 0.2
    if periodic:   # a periodic axis halves evenly down to the coarsest level
        nx = max(64, nx // 64 * 64)
    most = max(1, min(50, top // (nx * ny)))
    if kind == "restart":
        most = min(most, 10)
    steps = max(1, round(math.exp(rng.uniform(math.log(max(1.0, most / 4)), math.log(most)))))
    calls = rng.choice([1, 1, steps]) if steps <= 10 else 1
    return _case(kind, precision, nx, ny, steps=steps // calls, calls=calls, radius=rng.uniform(0.3, 0.42) * min(ny, 0.6 * nx),
                 periodic_x=periodic, mag_bc=rng.choice([0, 0, 0, 1]) if not periodic else 0,
                 autotune=nx >= 2048 and rng.random() < 0.5, **phys)


# ---- inputs ---------------------------------------------------------------------
def _descs(case):
    """the library's case descriptions"""
    if case["kind"] == "batch":
        return I.sweep_cases(case["ncase"])
    return [I.case(case["nx"], case["ny"], radius=case["radius"], field_angle_deg=case["angle"], bo_m=case["bo"],
                   stefan=case["ste"], chi_l=case["chi"], chi_s=case["chi"], contact_angle_deg=case["theta"],
                   dts=case["dts"], periodic_x=int(case["periodic_x"]), mag_bc=case["mag_bc"],
                   gravity=case["gravity"])]


def _device():
    return torch.device("cuda" if torch.cuda.is_available() else "cpu")


def _latent(d):
    return d["cp_l"] * (d["T_m"] - d["wall_T"][2]) / d["stefan"]


def _field_strength(d):
    return math.sqrt(d["bo_m"] * d["sigma"] / (2.0 * d["radius"]))


def _state(d, seed):
    """A state half-way through the freezing of case d: {field id: (ny, nx) float64 tensor}."""
    r = random.Random(seed)
    dev, f8 = _device(), torch.float64
    nx, ny, R, L = d["nx"], d["ny"], d["radius"], _latent(d)
    x = (torch.arange(nx, device=dev, dtype=f8) + 0.5)[None, :]
    y = (torch.arange(ny, device=dev, dtype=f8) + 0.5)[:, None]

    def smooth():   # a few long waves, in [-1, 1]
        f = 0.0
        for _ in range(3):
            kx, ky = 2 * math.pi * r.randint(0, 2) / nx, 2 * math.pi * r.randint(0, 2) / ny
            f = f + r.uniform(0.3, 1.0) / 3.0 * torch.cos(kx * x + ky * y + r.uniform(0, 2 * math.pi))
        return f

    rr = torch.sqrt((x - 0.5 * nx) ** 2 + y ** 2)
    th = torch.atan2(y, x - 0.5 * nx)
    rim = 1.0
    for m in (2, 4, 6):
        rim = rim + r.uniform(-0.01, 0.01) * torch.cos(m * th + r.uniform(-0.3, 0.3))
    C = 0.5 + 0.5 * torch.tanh(2.0 * (R * rim - rr) / d["xi"])
    front = R * r.uniform(0.1, 0.35) * (1.0 + 0.05 * torch.cos(2 * math.pi * x / nx * r.randint(1, 3) + r.uniform(0, 6)))
    warm = r.uniform(0.01, 0.05)
    T = torch.where(y < front, d["wall_T"][2] * (1.0 - y / front), warm * (1.0 - torch.exp(-(y - front) / (0.3 * R))))
    cpL = d["cp_g"] + C * (d["cp_l"] - d["cp_g"])
    liquid = (y + 0.5 - front).clamp(0.0, 1.0)   # of the cell row that the front crosses
    He = torch.where(C < 0.5, cpL * T + L, liquid * (cpL * T.clamp(min=0.0) + L) + (1 - liquid) * d["cp_s"] * T.clamp(max=0.0))
    _, Fl = _eq8(d, He, C)
    rho = _mix(1 - Fl, C, d["rho_s"], d["rho_l"], d["rho_g"])
    calm = torch.sin(math.pi * y / ny) * (1.0 if d["periodic_x"] else torch.sin(math.pi * x / nx))
    mx = 0.02 / 3.0 * rho * Fl * calm * smooth()
    my = 0.02 / 3.0 * rho * Fl * calm * smooth()
    p = d["sigma"] / R * C + 0.002 * smooth()
    a = d["field_angle_deg"] * math.pi / 180.0
    phi = -_field_strength(d) * (x * math.cos(a) + y * math.sin(a))
    one = torch.ones((ny, nx), device=dev, dtype=f8)
    return {I.PHI: phi * one, I.HE: He, I.P: p * one, I.C: C, I.MX: mx, I.MY: my, I.FSPREV: 1.0 - Fl}


def _pinned(*shape, dtype=torch.float64):
    return torch.empty(shape, dtype=dtype, pin_memory=torch.cuda.is_available())


def prepare(case, seed):
    descs = _descs(case)
    prec = lbfs.FP64 if case["precision"] == "fp64" else lbfs.MIXED
    s = lbfs.Solver(precision=prec, max_cases=len(descs), use_graph=bool(case["graph"]))
    ids = {"monitor": DERIVED, "pseudo": [I.PHI]}.get(case["kind"], STATE)
    bufs, first = [], None
    for k, d in enumerate(descs):
        s.set_case(k, d)
        f = _state(d, seed * 1009 + k)
        packed = _pinned(len(CHECKPOINT), d["ny"], d["nx"])
        for q, fid in enumerate(CHECKPOINT):
            packed[q].copy_(f[fid])
        if case["kind"] == "restart":
            first = packed
        else:
            s.set_fields_packed(k, CHECKPOINT, packed.numpy())
        bufs.append(_pinned(len(ids), d["ny"], d["nx"]))
    if case["autotune"]:
        s.autotune()
    out = None   # where the fields of all cases are gathered, or turned into 32 bits
    if prec == lbfs.MIXED or len(bufs) > 1:
        out = torch.empty((len(ids), sum(b[0].numel() for b in bufs)),
                          dtype=torch.float32 if prec == lbfs.MIXED else torch.float64)
    return dict(case=case, solver=s, ids=ids, bufs=bufs, first=first, out=out,
                dtype=np.float32 if prec == lbfs.MIXED else np.float64)


def _read(st):
    """the outputs of every case: {field name: array}"""
    s, ids, bufs, out = st["solver"], st["ids"], st["bufs"], st["out"]
    off = 0
    for k, b in enumerate(bufs):
        s.fields_into(k, ids, b.numpy())
        if out is not None:
            n = b[0].numel()
            out[:, off:off + n].copy_(b.view(len(ids), n))
            off += n
    src = bufs[0] if out is None else out
    return {I.FIELD_NAMES[f]: src[q].view(-1) for q, f in enumerate(ids)}


def _stats(st, stats):
    return {k: np.array([x[k] for x in stats], dtype=st["dtype"]) for k in STATS}


def run(st):
    case, s = st["case"], st["solver"]
    if case["kind"] == "monitor":
        diag, q = s.diagnostics(0)
        return {"diag": {k: np.array(v, dtype=st["dtype"]) for k, v in diag.items()}, "q_wall": q.astype(st["dtype"]),
                "fields": _read(st)}
    if case["kind"] == "pseudo":
        s.potential_pseudo_time(0, case["steps"], 0.2 / (1.0 + case["chi"]))
        return _read(st)
    if case["kind"] == "restart":
        s.set_fields_packed(0, CHECKPOINT, st["first"].numpy())
    for _ in range(case["calls"]):
        stats = s.step(case["steps"])
    return {"stats": _stats(st, stats), "fields": _read(st)}


def work(case):
    """Bytes: per step the evolved state (H_e 8 bytes; p, two momenta and C), the potential (8 bytes)
    and the lagged solid fraction, read once and written once; then the 64-bit fields handed over.  Operations:
    per face the nine surrounding points' three equilibria and the interface values (about 350),
    two faces a cell and 150 for the cell itself, three stages a step."""
    cells = sum(d["nx"] * d["ny"] for d in _descs(case))
    r = 8 if case["precision"] == "fp64" else 4
    n = case["steps"] * case["calls"]
    if case["kind"] == "pseudo":
        return {"bytes": cells * n * (8 + 8 + r), "flops": cells * n * 25}
    if case["kind"] == "monitor":
        return {"bytes": cells * (8 + 4 * r + 8 * len(DERIVED)), "flops": cells * 60}
    moved = n * 2 * (16 + 5 * r) + 8 * len(STATE) + (8 * len(CHECKPOINT) if case["kind"] == "restart" else 0)
    return {"bytes": cells * moved, "flops": cells * n * 3 * (2 * 350 + 150)}


# ---- the same step in 64 bits, in plain torch ----------------------------------
EDIR = [(0, 0), (1, 0), (0, 1), (-1, 0), (0, -1), (1, 1), (-1, 1), (-1, -1), (1, -1)]
WDIR = [4 / 9] + [1 / 9] * 4 + [1 / 36] * 4


def _mix(Fs, C, gs, gl, gg):
    return Fs * gs + (1 - Fs) * (C * gl + (1 - C) * gg)


def _eq8(d, He, C):
    """Eq. 8: temperature and liquid fraction"""
    cpL = d["cp_g"] + C * (d["cp_l"] - d["cp_g"])
    Tm, L = d["T_m"], _latent(d)
    Hs, Hl = d["cp_s"] * Tm, cpL * Tm + L
    solid, liquid = (C >= 0.5) & (He < Hs), (C < 0.5) | (He > Hl)
    Fl = torch.where(solid, torch.zeros_like(He), torch.where(liquid, torch.ones_like(He), (He - Hs) / (Hl - Hs)))
    T = torch.where(solid, He / d["cp_s"], torch.where(liquid, Tm + (He - Hl) / cpL, torch.full_like(He, Tm)))
    return T, Fl


class _Exact:
    """One case in 64 bits: the finite-volume update evaluated direction by direction, and the
    potential by conjugate gradients preconditioned with the constant-coefficient operator (FFT)."""

    def __init__(self, d, state):
        self.d = d
        self.W = [state[f].clone() for f in (I.HE, I.P, I.MX, I.MY, I.C)]
        self.phi, self.Fs = state[I.PHI].clone(), state[I.FSPREV].clone()
        self.t = 0.0
        a = d["field_angle_deg"] * math.pi / 180.0
        self.hx, self.hy = -_field_strength(d) * math.cos(a), -_field_strength(d) * math.sin(a)
        self.per = (bool(d["periodic_x"]), bool(d["periodic_y"]))
        self.dirichlet = (not self.per[0] and d["mag_bc"] == 0, not self.per[1])
        dev, f8 = self.phi.device, torch.float64
        self.x = torch.arange(d["nx"], device=dev, dtype=f8) + 0.5
        self.y = torch.arange(d["ny"], device=dev, dtype=f8) + 0.5
        self.wet = 0.0 if d["contact_angle_deg"] == 90.0 else 4.0 * math.cos(d["contact_angle_deg"] * math.pi / 180.0) / d["xi"]

    def pad(self, f, ghost):
        """f with one ghost layer; ghost(edge values, wall) on the walls 0 left, 1 right, 2 bottom, 3 top"""
        ny, nx = f.shape
        g = f.new_zeros((ny + 2, nx + 2))
        g[1:-1, 1:-1] = f
        g[1:-1, 0] = f[:, -1] if self.per[0] else ghost(f[:, 0], 0)
        g[1:-1, -1] = f[:, 0] if self.per[0] else ghost(f[:, -1], 1)
        g[0, 1:-1] = f[-1] if self.per[1] else ghost(f[0], 2)
        g[-1, 1:-1] = f[0] if self.per[1] else ghost(f[-1], 3)
        return g

    def wall_phi(self, w):
        nx, ny = self.d["nx"], self.d["ny"]
        return self.hx * (nx * (w == 1)) + self.hy * self.y if w < 2 else self.hx * self.x + self.hy * (ny * (w == 3))

    # the potential, Eq. 4
    def matvec(self, mu, v):
        out = torch.zeros_like(v)
        for dim in (1, 0):
            per, dirichlet = self.per[1 - dim], self.dirichlet[1 - dim]
            n = v.shape[dim]
            F = 0.5 * (mu.narrow(dim, 0, n - 1) + mu.narrow(dim, 1, n - 1)) * (v.narrow(dim, 0, n - 1) - v.narrow(dim, 1, n - 1))
            out.narrow(dim, 0, n - 1).add_(F)
            out.narrow(dim, 1, n - 1).sub_(F)
            a, b, ma, mb = v.select(dim, 0), v.select(dim, n - 1), mu.select(dim, 0), mu.select(dim, n - 1)
            if per:
                F = 0.5 * (ma + mb) * (b - a)
                out.select(dim, n - 1).add_(F)
                out.select(dim, 0).sub_(F)
            elif dirichlet:
                out.select(dim, 0).add_(2 * ma * a)
                out.select(dim, n - 1).add_(2 * mb * b)
        return out

    def precondition(self, r):
        ny, nx = r.shape
        if not hasattr(self, "lam"):
            lam = lambda n, per: 2 - 2 * torch.cos(2 * math.pi * torch.arange(n if per else 2 * n, device=r.device, dtype=r.dtype) / (n if per else 2 * n))  # noqa: E731
            lx = lam(nx, self.per[0])
            m = lx.numel()
            self.lam = lam(ny, self.per[1])[:, None] + lx[None, : m // 2 + 1]
            self.lam[self.lam == 0] = 1.0
        e = r
        if not self.per[0]:
            e = torch.cat([e, (-1 if self.dirichlet[0] else 1) * e.flip(1)], 1)
        if not self.per[1]:
            e = torch.cat([e, -e.flip(0)], 0)
        return torch.fft.irfft2(torch.fft.rfft2(e) / self.lam, s=e.shape)[:ny, :nx].contiguous()

    def solve_potential(self):
        d = self.d
        if (d["chi_l"] == d["chi_s"] == d["chi_g"] == 0.0) or not any(self.dirichlet):
            return
        _, Fl = _eq8(d, self.W[0], self.W[4])
        mu = 1.0 + _mix(1 - Fl, self.W[4], d["chi_s"], d["chi_l"], d["chi_g"])
        b = torch.zeros_like(mu)
        for dim in (1, 0):
            if self.dirichlet[1 - dim]:
                lo, hi = (0, 1) if dim == 1 else (2, 3)
                b.select(dim, 0).add_(2 * mu.select(dim, 0) * self.wall_phi(lo))
                b.select(dim, -1).add_(2 * mu.select(dim, -1) * self.wall_phi(hi))
        small = 3e-15 * float(b.norm())
        r = b - self.matvec(mu, self.phi)
        z = self.precondition(r)
        p, rz = z, torch.sum(r * z)
        for _ in range(60):
            if float(r.norm()) <= small:
                break
            q = self.matvec(mu, p)
            alpha = rz / torch.sum(p * q)
            self.phi = self.phi + alpha * p
            r = r - alpha * q
            z = self.precondition(r)
            new = torch.sum(r * z)
            p, rz = z + (new / rz) * p, new

    def field2(self):
        """|H|^2 with its ghost layer"""
        ph = self.pad(self.phi, lambda e, w: 2 * self.wall_phi(w) - e if self.dirichlet[w // 2] else e)
        hx, hy = 0.5 * (ph[1:-1, 2:] - ph[1:-1, :-2]), 0.5 * (ph[2:, 1:-1] - ph[:-2, 1:-1])
        return self.pad(hx * hx + hy * hy, lambda e, w: e)

    def muc(self, Cg):
        d, C = self.d, Cg[1:-1, 1:-1]
        beta, kappa = 12.0 * d["sigma"] / d["xi"], 1.5 * d["xi"] * d["sigma"]
        lap = Cg[1:-1, 2:] + Cg[1:-1, :-2] + Cg[2:, 1:-1] + Cg[:-2, 1:-1] - 4 * C
        return 2 * beta * C * (C - 1) * (2 * C - 1) - kappa * lap

    def wetted(self, C):
        return self.pad(C, lambda e, w: e + self.wet * e * (1 - e))

    def faces(self, dim, q, grad_n, grad_t, Fs):
        """fluxes of the interior faces across dim: (H_e, p, normal and tangential momentum, C)"""
        d, dts = self.d, self.d["dts"]
        n = Fs.shape[dim]
        per = self.per[1 - dim]
        A = (lambda f: f.roll(1, dim)) if per else (lambda f: f.narrow(dim, 0, n - 1))
        B = (lambda f: f) if per else (lambda f: f.narrow(dim, 1, n - 1))
        fsA, fsB = A(Fs), B(Fs)
        fsm = 0.5 * (fsA + fsB)
        cpref, Qg = 0.5 * (d["cp_s"] + d["cp_l"]), d["Q_g"]
        sums = [0.0] * 5          # f, e_n f, e_t f, g, h
        en_g = en_h = p_nn = p_nt = gam_nn = gam_nt = 0.0
        for (en, et), w in zip(EDIR, WDIR):
            vals = []
            for f, gn, gt in zip(q, grad_n, grad_t):
                va = A(f) + (0.5 - en * dts) * A(gn) - et * dts * A(gt) if en >= 0 else None
                vb = B(f) + (-0.5 - en * dts) * B(gn) - et * dts * B(gt) if en <= 0 else None
                vals.append(va if vb is None else vb if va is None else 0.5 * (va + vb))
            p, un, ut, C, m, T, H = vals
            fs = fsA if en > 0 else fsB if en < 0 else fsm
            rho, cp = _mix(fs, C, d["rho_s"], d["rho_l"], d["rho_g"]), _mix(fs, C, d["cp_s"], d["cp_l"], d["cp_g"])
            eu = en * un + et * ut
            gam = 3 * eu + 4.5 * eu * eu - 1.5 * (un * un + ut * ut)
            feq = w * (p + rho / 3 * gam)
            if en == 0 and et == 0:
                geq = C - 5 / 3 * m * Qg
                heq = H - cpref * T + w * T * (cpref + cp * gam)
            else:
                geq = 3 * w * (m * Qg + C * eu)
                heq = w * T * (cpref + cp * gam)
            for k, v in enumerate((feq, en * feq, et * feq, geq, heq)):
                sums[k] = sums[k] + v
            en_g, en_h = en_g + en * geq, en_h + en * heq
            p_nn, p_nt = p_nn + en * en * w * p, p_nt + en * et * w * p
            gam_nn, gam_nt = gam_nn + en * en * w * gam, gam_nt + en * et * w * gam
        pf, jn, jt, Cf, Hf = sums
        rho = _mix(fsm, Cf, d["rho_s"], d["rho_l"], d["rho_g"])
        un, ut = 3 * jn / rho, 3 * jt / rho
        cp = _mix(fsm, Cf, d["cp_s"], d["cp_l"], d["cp_g"])
        lam = _mix(fsm, Cf, d["lam_s"], d["lam_l"], d["lam_g"])
        mu = _mix(fsm, Cf, d["mu_s"], d["mu_l"], d["mu_g"])
        Tf, _ = _eq8(d, Hf, Cf)
        tf, th, tg = 0.5 + 3 * mu / (rho * dts), 0.5 + 3 * lam / (rho * cpref * dts), 0.5 + d["mobility"] / (Qg * dts)
        Fh = (1.5 - th) * cp * Tf * un + (th - 0.5) * en_h
        Fc = (1.5 - tg) * Cf * un + (tg - 0.5) * en_g
        Fn = (1.5 - tf) / 3 * (pf + rho * un * un) + (tf - 0.5) * (p_nn + rho / 3 * gam_nn)
        Ft = (1.5 - tf) / 3 * rho * un * ut + (tf - 0.5) * (p_nt + rho / 3 * gam_nt)
        return Fh, jn, Fn, Ft, Fc

    def wall(self, w, at, q, Fs, rho):
        """the flux of wall w, from its row of inner cells"""
        d = self.d
        p, u, v, C, _, T, _ = (at(f) for f in q)
        fs = at(Fs)
        mu, lam = _mix(fs, C, d["mu_s"], d["mu_l"], d["mu_g"]), _mix(fs, C, d["lam_s"], d["lam_l"], d["lam_g"])
        side = 1.0 if w in (0, 2) else -1.0
        ut = v if w < 2 else u
        heat = -lam / at(rho) * side * 2 * (T - d["wall_T"][w]) if d["thermal_dirichlet"][w] else torch.zeros_like(T)
        zero = torch.zeros_like(T)
        return heat, zero, p / 3, -mu * side * 2 * ut / 3, zero

    def rhs(self, W, H2, Sd):
        d = self.d
        He, p, mx, my, C = W
        T, Fl = _eq8(d, He, C)
        Fs, L = 1 - Fl, _latent(d)
        rho = _mix(Fs, C, d["rho_s"], d["rho_l"], d["rho_g"])
        cp = _mix(Fs, C, d["cp_s"], d["cp_l"], d["cp_g"])
        u, v = 3 * mx / rho, 3 * my / rho
        same, odd = (lambda e, w: e), (lambda e, w: -e)
        Cg = self.wetted(C)
        m = self.muc(Cg)
        edge = {0: (slice(None), 0), 1: (slice(None), -1), 2: (0,), 3: (-1,)}
        Tw = lambda e, w: 2 * d["wall_T"][w] - e if d["thermal_dirichlet"][w] else e  # noqa: E731
        Hw = lambda e, w: cp[edge[w]] * Tw(T[edge[w]], w) + L * Fl[edge[w]]  # noqa: E731
        q = [p, u, v, C, m, T, He]
        padded = [self.pad(p, same), self.pad(u, odd), self.pad(v, odd), Cg, self.pad(m, same), self.pad(T, Tw), self.pad(He, Hw)]
        gx = [0.5 * (g[1:-1, 2:] - g[1:-1, :-2]) for g in padded]
        gy = [0.5 * (g[2:, 1:-1] - g[:-2, 1:-1]) for g in padded]
        rg = self.pad(rho, same)
        R = [torch.zeros_like(C) for _ in range(5)]
        for dim in (1, 0):
            order = [0, 1, 2, 3, 4, 5, 6] if dim == 1 else [0, 2, 1, 3, 4, 5, 6]
            n, t = (gx, gy) if dim == 1 else (gy, gx)
            F = self.faces(dim, [q[k] for k in order], [n[k] for k in order], [t[k] for k in order], Fs)
            if self.per[1 - dim]:
                F = [torch.cat([f, f.narrow(dim, 0, 1)], dim) for f in F]
            else:
                lo, hi = (0, 1) if dim == 1 else (2, 3)
                a = self.wall(lo, lambda f: f.select(dim, 0), q, Fs, rho)
                b = self.wall(hi, lambda f: f.select(dim, -1), q, Fs, rho)
                F = [torch.cat([x.unsqueeze(dim), f, y.unsqueeze(dim)], dim) for x, f, y in zip(a, F, b)]
            size = C.shape[dim]
            to = (0, 1, 2, 3, 4) if dim == 1 else (0, 1, 3, 2, 4)
            for k, f in zip(to, F):
                R[k] -= f.narrow(dim, 1, size) - f.narrow(dim, 0, size)
        chi = _mix(Fs, C, d["chi_s"], d["chi_l"], d["chi_g"])
        vr = 1.0 - d["rho_s"] / d["rho_l"]
        cx, cy = (lambda g: 0.5 * (g[1:-1, 2:] - g[1:-1, :-2])), (lambda g: 0.5 * (g[2:, 1:-1] - g[:-2, 1:-1]))
        R[0] += cp * T * (gx[1] + gy[2])
        R[1] += (u * cx(rg) + v * cy(rg)) / 3 + rho / 3 * vr * Sd
        R[2] += (-C * gx[4] + 0.5 * chi * cx(H2) - rho * u * Sd) / 3
        R[3] += (-C * gy[4] + 0.5 * chi * cy(H2) + rho * d["gravity"] - rho * v * Sd) / 3
        R[4] += C * vr * Sd
        return R

    def step(self):
        d = self.d
        dt = d["dt"]
        _, Fl = _eq8(d, self.W[0], self.W[4])
        Sd, self.Fs = ((1 - Fl) - self.Fs) / dt, 1 - Fl
        self.solve_potential()
        H2 = self.field2()
        W0, W = self.W, self.W
        for a, b in ((0.0, 1.0), (0.75, 0.25), (1.0 / 3.0, 2.0 / 3.0)):
            W = [a * w0 + b * (w + dt * r) for w0, w, r in zip(W0, W, self.rhs(W, H2, Sd))]
        _, Fl = _eq8(d, W[0], W[4])
        W[2], W[3] = W[2] * Fl, W[3] * Fl
        self.W = W
        self.t += dt

    def out(self):
        return dict(zip((I.HE, I.P, I.MX, I.MY, I.C, I.PHI), self.W + [self.phi]))

    def stats(self):
        He, C = self.W[0], self.W[4]
        _, Fl = _eq8(self.d, He, C)
        drop = C >= 0.5
        n = float(drop.sum())
        return {"sum_C": float(C.sum()), "sum_He": float(He.sum()), "sum_Fl_drop": float(Fl[drop].sum()), "n_drop": n,
                "Q_L": float((1 - Fl)[drop].sum()) / max(n, 1.0), "t": self.t}

    # Sec. 5 diagnostics and derived fields
    def derived(self):
        d = self.d
        He, _, mx, my, C = self.W
        T, Fl = _eq8(d, He, C)
        rho = _mix(1 - Fl, C, d["rho_s"], d["rho_l"], d["rho_g"])
        return {I.T: T, I.FL: Fl, I.U: 3 * mx / rho, I.V: 3 * my / rho, I.MUC: self.muc(self.wetted(C)), I.RHO: rho}

    def diagnostics(self):
        d = self.d
        f, C = self.derived(), self.W[4]
        ny = d["ny"]
        drop = C >= 0.5
        top = ny - 1 - drop.flip(0).to(torch.int64).argmax(0)
        some = drop.any(0)
        c0 = C.gather(0, top[None])[0]
        c1 = C.gather(0, (top + 1).clamp(max=ny - 1)[None])[0]
        h = torch.where(top == ny - 1, torch.full_like(c0, float(ny)), top + 0.5 + (c0 - 0.5) / (c0 - c1))
        H_m = float(torch.where(some, h, torch.zeros_like(h)).max())
        U = float((torch.sqrt(f[I.U] ** 2 + f[I.V] ** 2) * drop).max())
        lam = _mix(1 - f[I.FL][0], C[0], d["lam_s"], d["lam_l"], d["lam_g"])
        q = -lam * (-8 * d["wall_T"][2] + 9 * f[I.T][0] - f[I.T][1]) / 3
        alpha, R0 = d["lam_l"] / (d["rho_l"] * d["cp_l"]), d["radius"]
        return {"H_m": H_m, "U_max": U, "Pe": U * 2 * R0 / alpha, "Fo": alpha * self.t / (R0 * R0), "Q_wall": float(q.sum())}, q

    def pseudo_time(self, n, dtau):
        """n explicit steps of the pseudo-time relaxation with the magnetic face flux"""
        d = self.d
        _, Fl = _eq8(d, self.W[0], self.W[4])
        mu = 1.0 + _mix(1 - Fl, self.W[4], d["chi_s"], d["chi_l"], d["chi_g"])
        dts = d["dts"]
        for _ in range(n):
            ph = self.pad(self.phi, lambda e, w: 2 * self.wall_phi(w) - e if self.dirichlet[w // 2] else e)
            div = torch.zeros_like(mu)
            for dim in (1, 0):
                size = mu.shape[dim]
                grad = 0.5 * (ph[1:-1, 2:] - ph[1:-1, :-2] if dim == 1 else ph[2:, 1:-1] - ph[:-2, 1:-1])
                a, b = (lambda f: f.narrow(dim, 0, size - 1)), (lambda f: f.narrow(dim, 1, size - 1))
                F = 0.5 * (a(mu) + b(mu)) / (2 * dts) * (a(self.phi) - b(self.phi) + (0.5 - dts) * (a(grad) + b(grad)))
                div.narrow(dim, 0, size - 1).add_(F)
                div.narrow(dim, 1, size - 1).sub_(F)
                if self.dirichlet[1 - dim]:
                    lo, hi = (0, 1) if dim == 1 else (2, 3)
                    div.select(dim, 0).add_(2 * mu.select(dim, 0) * (self.phi.select(dim, 0) - self.wall_phi(lo)))
                    div.select(dim, -1).add_(2 * mu.select(dim, -1) * (self.phi.select(dim, -1) - self.wall_phi(hi)))
            self.phi = self.phi - dtau * div


def exact(case, seed):
    descs = _descs(case)
    n = case["steps"] * case["calls"]
    if case["kind"] == "batch" and len(descs) * n > 1300:
        return None   # several minutes
    done = []
    for k, d in enumerate(descs):
        e = _Exact(d, _state(d, seed * 1009 + k))
        if case["kind"] == "pseudo":
            e.pseudo_time(n, 0.2 / (1.0 + case["chi"]))
        elif case["kind"] != "monitor":
            for _ in range(n):
                e.step()
        done.append(e)
    if case["kind"] == "monitor":
        diag, q = done[0].diagnostics()
        f = done[0].derived()
        return {"diag": {k: np.array(v) for k, v in diag.items()}, "q_wall": q, "fields": {I.FIELD_NAMES[i]: f[i].reshape(-1) for i in DERIVED}}
    if case["kind"] == "pseudo":
        return {I.FIELD_NAMES[I.PHI]: done[0].phi.reshape(-1)}
    stats = [e.stats() for e in done]
    outs = [e.out() for e in done]
    return {"stats": {k: np.array([s[k] for s in stats]) for k in STATS},
            "fields": {I.FIELD_NAMES[i]: torch.cat([o[i].reshape(-1) for o in outs]) for i in STATE}}

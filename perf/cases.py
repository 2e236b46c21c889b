"""What this package is used for, as cases that can be timed and checked.

Every case goes through the public entry points (``egpe.py``, ``autograd.py``) on
the grids and couplings of ``inputs.PRESETS`` and of the parameter scan: single
evaluations (energy/gradient, line-search coefficients, preconditioner), solver
runs cut after a fixed number of iterations (NCG in FP64, FP32 and mixed
precision, the batched scan, imaginary-time evolution) and the differentiable
energy, forward and backward.

Results of FP32 fields are returned in 32 bits, scalars included: a handle with
FP32 fields (and a mixed solve that is cut short of convergence) reports its
energies as FP64 numbers, but they are as accurate as its fields.
"""
import math

import numpy as np
import torch

from paper_2510_24543_gb300 import autograd as A
from paper_2510_24543_gb300 import egpe as E
from paper_2510_24543_gb300 import inputs as I

SIZES = (16, 32, 48, 64, 80, 96, 128, 256)
SCAN_SIZES = (48, 64, 80, 96)
PREC = {"fp64": E.EGPE_FP64, "fp32": E.EGPE_FP32, "mixed": E.EGPE_MIXED}
PRECOND = {"none": 0, "kinetic": 1, "diagonal": 2, "kinetic+diagonal": 3, "blend": 4}


def listed():
    def case(name, op, prec, n, physics, **kw):
        return dict(name=name, op=op, prec=prec, nx=n[0], ny=n[1], nz=n[2], physics=physics, **kw)

    return [
        # the smallest call: one energy/gradient evaluation inside a caller's own optimiser
        case("energy-grad 32^3 fp64", "energy_grad", "fp64", (32, 32, 32), "c1"),
        # the plain FP64 workload: a whole small solve, where launches and polls count
        case("ncg 32^3 fp64", "ncg", "fp64", (32, 32, 32), "c1", precond="kinetic", iters=8),
        # a caller's own line search on the droplet grid
        case("line-coeffs 64^3 fp64", "line_coeffs", "fp64", (64, 64, 64), "c2"),
        # the droplet workload, both preconditioners
        case("ncg 64^3 fp64", "ncg", "fp64", (64, 64, 64), "c2", precond="kinetic+diagonal", iters=8),
        # the paper's baseline method on the same grid
        case("ite 64^3 fp64", "ite", "fp64", (64, 64, 64), "c2", iters=4, dtau=1e-3),
        # uneven mixed-radix grid: the preconditioner of a caller's own iteration
        case("precondition 80x96x48 fp32", "precondition", "fp32", (80, 96, 48), "c2", precond="kinetic+diagonal"),
        # the headline workload, FP32 fields
        case("ncg 128^3 fp32", "ncg", "fp32", (128, 128, 128), "c3p", precond="kinetic+diagonal", iters=12),
        # the same in plain FP64
        case("ncg 128^3 fp64", "ncg", "fp64", (128, 128, 128), "c3p", precond="kinetic+diagonal", iters=3),
        # the stripe/supersolid workload in mixed precision: FP32 phase, then FP64 polish
        case("ncg 128x128x64 mixed", "ncg", "mixed", (128, 128, 64), "c3", precond="kinetic+diagonal", iters=2,
             iters_fp32=8),
        # the parameter scan: uneven grids advanced together, 4 instances of each
        case("scan 48^3..96^3 mixed", "scan", "mixed", (48, 48, 96), "scan", precond="kinetic+diagonal", iters=2,
             iters_fp32=8, count=16),
        # the differentiable large solve's step: energy forward, psi and parameter gradients backward
        case("autograd 256x256x128 fp32", "autograd", "fp32", (256, 256, 128), "c5"),
        # the largest evaluation
        case("energy-grad 256x256x128 fp64", "energy_grad", "fp64", (256, 256, 128), "c5"),
    ]


# grid points times iterations that a drawn case may ask for (the listed ones' largest per kind)
LIMIT = {"fp64": 3 * 128 ** 3, "fp32": 12 * 128 ** 3, "mixed": 3 * 128 ** 3}


def draw(rng):
    op = rng.choice(["energy_grad", "line_coeffs", "precondition", "ncg", "ncg", "ncg", "scan", "ite", "autograd"])
    prec = rng.choice(["fp64", "fp32", "mixed"] if op in ("ncg", "scan") else ["fp64", "fp32"])
    c = dict(op=op, prec=prec, nx=48, ny=48, nz=96, physics=rng.choice(["c1", "c2", "c3p", "c5"]),
             sample=rng.randrange(1 << 20))
    if op in ("ncg", "scan"):
        c["precond"] = rng.choice(["kinetic", "kinetic+diagonal", "kinetic+diagonal", "diagonal", "blend", "none"])
        # FP32 fields: long runs with both preconditioners, as the workloads have it; the other modes
        # approach the minimum along soft modes, where a run's rounding grows with every iteration
        c["iters"] = rng.randrange(2, 9) if prec == "fp64" or c["precond"] == "kinetic+diagonal" else rng.randrange(1, 3)
        if prec == "mixed":
            c["iters_fp32"], c["iters"] = c["iters"], rng.randrange(1, 4)
    elif op == "ite":
        c.update(iters=rng.randrange(2, 6), dtau=1e-3)
    elif op == "precondition":
        c["precond"] = rng.choice(["kinetic", "kinetic+diagonal", "kinetic+diagonal", "blend"])
    if op == "scan":
        c.update(physics="scan", count=4 * rng.randrange(1, 5))
        c["iters"] = min(c["iters"], 8 if prec == "fp32" else 2)
        return c
    most = LIMIT[prec] // max(1, c.get("iters", 1)) if op in ("ncg", "ite") else 256 * 256 * 128
    want = math.exp(rng.uniform(math.log(16 ** 3), math.log(most)))
    tries = [tuple(rng.choice(SIZES) for _ in range(3)) for _ in range(60)]
    tries = [n for n in tries if n[0] * n[1] * n[2] <= most] or [(32, 32, 32)]
    c["nx"], c["ny"], c["nz"] = min(tries, key=lambda n: abs(math.log(n[0] * n[1] * n[2] / want)))
    return c


def _workloads(case):
    """The case's instances.  Drawn cases ("sample") vary the couplings over the scan's range."""
    if case["op"] == "scan":
        w = I.scan_workloads(64, 4242 + case.get("sample", 0))
        per = case["count"] // len(SCAN_SIZES)
        return [w[16 * s + k] for s in range(len(SCAN_SIZES)) for k in range(per)]
    b = I.PRESETS[case["physics"]]
    g, gdd = b.g, b.gdd
    if "sample" in case:
        s = I.scan_workloads(64, 4242 + case["sample"])[case["sample"] % 64]
        g12 = 0.5 * (g[0][0] + g[1][1]) * s.g[0][1] / s.g[0][0]
        g, gdd = ((g[0][0], g12), (g12, g[1][1])), tuple(tuple(0.8 * s.gdd[0][0] for _ in range(2)) for _ in range(2))
    return [I.Workload(b.name, (case["nx"], case["ny"], case["nz"]), b.L, b.trap, g, gdd, b.lhy_c, b.seed, b.precond)]


def _grid(w):
    """Coordinates (z, y, x, broadcastable) and dV on the GPU."""
    xs = [torch.from_numpy(a).cuda() for a in I.axes(w.n, w.L)]
    dV = math.prod(2.0 * w.L[a] / w.n[a] for a in range(3))
    return xs[2][:, None, None], xs[1][None, :, None], xs[0][None, None, :], dV


def _unit(psi, dV):
    return psi / torch.sqrt(dV * psi.abs().square().sum(dim=(1, 2, 3), keepdim=True))


def _start(w, seed, phase):
    """The trap's Gaussian times 1 + 1% noise (the workloads' start); with `phase`, a state
    inside a run of a complex problem: complex noise and a smooth phase."""
    z, y, x, dV = _grid(w)
    gen = torch.Generator(device="cuda").manual_seed(seed)
    env = torch.exp(-0.5 * (w.trap[0] * x ** 2 + w.trap[1] * y ** 2 + w.trap[2] * z ** 2))
    shape = (2, w.n[2], w.n[1], w.n[0])
    noise = torch.randn(shape, generator=gen, device="cuda", dtype=torch.float64)
    psi = (env * (1.0 + 0.01 * noise)).to(torch.complex128)
    if phase:
        noise = torch.randn(shape, generator=gen, device="cuda", dtype=torch.float64)
        psi = psi + 0.01j * env * noise
        psi = psi * torch.exp(1j * (0.3 * torch.sin(2 * x / w.L[0]) + 0.2 * torch.cos(y / w.L[1] + z / w.L[2])))
    return _unit(psi, dV)


def _direction(w, psi):
    """A descent direction as a caller's optimiser has it: -V psi with a smooth modulation, made tangent."""
    z, y, x, dV = _grid(w)
    V = 0.5 * ((w.trap[0] * x) ** 2 + (w.trap[1] * y) ** 2 + (w.trap[2] * z) ** 2)
    d = -(V / (1.0 + V)) * psi * (1.0 + 0.2j * torch.sin(x / w.L[0]))
    c = dV * (d.conj() * psi).sum(dim=(1, 2, 3), keepdim=True).real
    return (d - c * psi).contiguous()


def _inputs(case, seed):
    """[(workload, psi in FP64, as the handle's fields hold it)]."""
    ws = _workloads(case)
    out = []
    for k, w in enumerate(ws):
        psi = _start(w, (1000003 * k + seed) & 0x7FFFFFFF, case["op"] not in ("ncg", "scan", "ite"))
        if case["prec"] == "fp32":
            psi = psi.to(torch.complex64)
        out.append((w, psi.contiguous()))
    return out


class _Handle:
    def __init__(self, ws, prec):
        self.h = E.egpe_create([E.make_grid(w.n, w.L) for w in ws], [E.params_from_workload(w) for w in ws], prec)

    def __del__(self):
        E.egpe_destroy(self.h)


def _opts(case):
    o = E.egpe_default_solve_opts()
    o.precond = PRECOND[case["precond"]]
    o.tol_res = 0.0  # a fixed number of iterations
    o.tol_fp32_switch = 0.0
    o.max_iter = case["iters"]
    o.max_iter_fp32 = case.get("iters_fp32", 0)
    return o


def prepare(case, seed):
    ins = _inputs(case, seed)
    w, psi = ins[0]
    s = dict(case=case, psi=[p for _, p in ins])
    if case["op"] == "autograd":
        s["theta"] = A.params_vector(w.g, w.gdd, w.kappa, w.eta_s, w.trap).requires_grad_(True)
        s["model"] = A.EnergyModel(w.n, w.L, s["theta"], w.lhy_nodes, PREC[case["prec"]])
        psi.requires_grad_(True)
        return s
    s["handle"] = _Handle([x for x, _ in ins], PREC[case["prec"]])
    if case["op"] in ("energy_grad", "precondition"):
        s["out"] = torch.empty_like(psi)
    if case["op"] == "line_coeffs":
        s["p"] = _direction(w, psi.to(torch.complex128)).to(psi.dtype)
    if case["op"] in ("ncg", "scan", "ite"):
        s["x"] = [torch.empty_like(p) for p in s["psi"]]
    if case["op"] in ("ncg", "scan"):
        s["opts"] = _opts(case)
    if case["op"] == "ite":
        o = E.egpe_default_ite_opts()
        o.dtau, o.tol_dE, o.max_steps = case["dtau"], 1e-30, case["iters"]
        s["opts"] = o
    return s


def _scalars(case, *v):
    return list(v) if case["prec"] == "fp64" else [np.float32(x) for x in v]


def run(s):
    case, op = s["case"], s["case"]["op"]
    if op == "autograd":
        psi, theta = s["psi"][0], s["theta"]
        e = s["model"].energy(psi, theta)
        g_psi, g_theta = torch.autograd.grad(e, (psi, theta))
        return [e, g_psi, g_theta] if case["prec"] == "fp64" else [e.float(), g_psi, g_theta.float()]
    h = s["handle"].h
    if op == "energy_grad":
        e, mu = E.egpe_energy_grad(h, 0, s["psi"][0], s["out"])
        return [s["out"]] + _scalars(case, e, *mu)
    if op == "line_coeffs":
        return _scalars(case, *E.egpe_line_coeffs(h, 0, s["psi"][0], s["p"]))
    if op == "precondition":
        E.egpe_precondition(h, 0, PRECOND[case["precond"]], s["psi"][0], None, s["out"])
        return [s["out"]]
    for x, p in zip(s["x"], s["psi"]):
        x.copy_(p)  # the solvers work in place
    if op == "ite":
        _, reps = E.egpe_ite_solve(h, s["x"], s["opts"], len(s["x"]))
    else:
        _, reps, _ = E.egpe_ncg_solve(h, s["x"], s["opts"], len(s["x"]))
    out = []
    for x, r in zip(s["x"], reps):
        x = x.to(torch.complex64) if case["prec"] == "mixed" else x
        out.append([x] + _scalars(case, r["E"], *r["mu"]))
    return out


def work(case):
    """Inputs read once, outputs written once; flops: the transforms (5 N log2 N each) the method names
    and about 150 operations per point and evaluation."""
    by = fl = 0.0
    for w in _workloads(case):
        N, lg = w.points, math.log2(w.points)
        c = 8 if case["prec"] == "fp32" else 16
        by += 4 * c * N  # two fields in (four for the line search, which writes none), two out
        fft = 5.0 * N * lg
        evals = {"energy_grad": 6, "line_coeffs": 10, "precondition": 10, "autograd": 8}
        if case["op"] in evals:
            fl += evals[case["op"]] * fft + 300.0 * N
        elif case["op"] == "ite":
            fl += case["iters"] * (20 * fft + 400.0 * N)
        else:
            per = 14 if case["precond"] not in ("none", "diagonal") else 10
            fl += (case["iters"] + case.get("iters_fp32", 0)) * (per * fft + 400.0 * N) + 6 * fft
    return {"bytes": by, "flops": fl}


# ----------------------------------------------------------------------------
# The same quantities in 64 bits with plain torch
# ----------------------------------------------------------------------------
class _Plain:
    def __init__(self, w):
        self.w = w
        self.z, self.y, self.x, self.dV = _grid(w)
        k = []
        for a in range(3):
            j = np.arange(w.n[a])
            k.append(torch.from_numpy((np.pi / w.L[a]) * np.where(j < w.n[a] // 2, j, j - w.n[a])).cuda())
        kx, ky, kz = k[0][None, None, :], k[1][None, :, None], k[2][:, None, None]
        self.k2 = kx ** 2 + ky ** 2 + kz ** 2
        self.kdd = torch.where(self.k2 > 0, 3.0 * kz ** 2 / torch.where(self.k2 > 0, self.k2, 1.0) - 1.0, 0.0)
        self.V = 0.5 * ((w.trap[0] * self.x) ** 2 + (w.trap[1] * self.y) ** 2 + (w.trap[2] * self.z) ** 2)
        t, q = np.polynomial.legendre.leggauss(w.lhy_nodes)
        self.c5 = w.kappa * w.eta_s ** -2.5
        self.nodes = [(3.0 * (0.5 * (a + 1.0)) ** 2 - 1.0, self.c5 * 0.5 * b) for a, b in zip(t, q)]

    def dot(self, a, b):
        """Re <a_i, b_i> of both components."""
        return self.dV * (a.real * b.real + a.imag * b.imag).sum(dim=(1, 2, 3)) if a.is_complex() else \
            self.dV * (a * b).sum(dim=(1, 2, 3))

    def kin(self, f, mult):
        return torch.stack([torch.fft.ifftn(mult[i] * torch.fft.fftn(f[i])) for i in range(2)])

    def dip(self, n):
        g = self.w.gdd
        src = [g[i][0] * n[0] + g[i][1] * n[1] for i in range(2)]
        return torch.stack([torch.fft.ifftn(self.kdd * torch.fft.fftn(s)).real for s in src])

    def branches(self, n):
        for x, W in self.nodes:
            e = [[self.w.g[i][j] + self.w.gdd[i][j] * x for j in range(2)] for i in range(2)]
            d = e[0][0] * n[0] - e[1][1] * n[1]
            s = torch.sqrt(d * d + 4.0 * e[0][1] ** 2 * n[0] * n[1])
            rs = torch.where(s > 0, 1.0 / torch.where(s > 0, s, 1.0), 0.0)
            A = e[0][0] * n[0] + e[1][1] * n[1]
            yield x, W, e, d, s, rs, (A + s).clamp_min(0.0), (A - s).clamp_min(0.0)

    def lhy(self, n, eta=False):
        """mu_LHY, the density F and, with `eta`, the integrals of its derivatives in (g11, g12, g22, gdd..)."""
        F, m1, m2 = (torch.zeros_like(n[0]) for _ in range(3))
        d6 = [0.0] * 6
        for x, W, e, d, s, rs, vp, vm in self.branches(n):
            F += W * (vp ** 2.5 + vm ** 2.5)
            sig1 = (e[0][0] * d + 2.0 * e[0][1] ** 2 * n[1]) * rs
            sig2 = (-e[1][1] * d + 2.0 * e[0][1] ** 2 * n[0]) * rs
            fp, fm = 2.5 * W * vp ** 1.5, 2.5 * W * vm ** 1.5
            m1 += fp * (e[0][0] + sig1) + fm * (e[0][0] - sig1)
            m2 += fp * (e[1][1] + sig2) + fm * (e[1][1] - sig2)
            if eta:
                t = [((fp + fm) * n[0] + (fp - fm) * d * n[0] * rs), (fp - fm) * 4.0 * e[0][1] * n[0] * n[1] * rs,
                     ((fp + fm) * n[1] - (fp - fm) * d * n[1] * rs)]
                for k in range(3):
                    v = self.dV * t[k].sum()
                    d6[k] += v
                    d6[3 + k] += x * v
        return torch.stack([m1, m2]), F, d6

    def point(self, psi):
        w, n = self.w, psi.abs().square()
        T, Phi = self.kin(psi, [0.5 * self.k2] * 2), self.dip(n)
        muL, F, _ = self.lhy(n)
        gn = torch.stack([w.g[i][0] * n[0] + w.g[i][1] * n[1] for i in range(2)])
        U = self.V + gn + Phi + muL
        H = T + U * psi
        e = self.dot(psi, T).sum() + self.dV * ((self.V * n).sum() + 0.5 * (n * (gn + Phi)).sum() + F.sum())
        mu = self.dot(psi, H)
        return dict(psi=psi, n=n, E=float(e), mu=mu, H=H, U=U, PV=self.V + gn + muL,
                    shift=(mu - self.dot(n, Phi)).abs())

    def precondition(self, pt, r, mode):
        a = pt["shift"][:, None, None, None]
        PV = torch.maximum(a + pt["PV"], 1e-2 * a)
        PD = [1.0 / (a[i] + 0.5 * self.k2) for i in range(2)]
        if mode == "none":
            return r
        if mode == "diagonal":
            return r / PV
        if mode == "blend":
            return 0.5 * r / PV + 0.5 * self.kin(r, PD)
        return self.kin(r / PV if mode == "kinetic+diagonal" else r, PD)

    def line(self, pt, p):
        """E', E'' along the geodesic."""
        w, psi, n = self.w, pt["psi"], pt["n"]
        rho = (psi.conj() * p).real
        a = p.abs().square()
        Pr = self.dip(rho)
        Ep = 2.0 * self.dot(p, pt["H"]).sum()
        Epp = 2.0 * (-self.dot(p, p) * pt["mu"] + self.dot(p, self.kin(p, [0.5 * self.k2] * 2))
                     + self.dot(pt["U"], a)).sum()
        gr = torch.stack([w.g[i][0] * rho[0] + w.g[i][1] * rho[1] for i in range(2)])
        Epp = Epp + 4.0 * self.dot(rho, gr + Pr).sum()
        n1p, n2p = 2.0 * rho[0], 2.0 * rho[1]
        h = torch.zeros_like(n1p)
        for x, W, e, d, s, rs, vp, vm in self.branches(n):
            d1 = e[0][0] * n1p - e[1][1] * n2p
            t1 = (d * d1 + 2.0 * e[0][1] ** 2 * (n[0] * n2p + n1p * n[1])) * rs
            K = (d1 * d1 + 4.0 * e[0][1] ** 2 * n1p * n2p - t1 * t1) * (0.5 * rs)
            A1 = e[0][0] * n1p + e[1][1] * n2p
            h += 2.5 * W * (2.0 * K * (vp ** 1.5 - vm ** 1.5)
                            + 1.5 * (vp ** 0.5 * (A1 + t1) ** 2 + vm ** 0.5 * (A1 - t1) ** 2))
        return float(Ep), float(Epp + self.dV * h.sum())

    def ncg(self, psi, mode, iters, tau):
        pt, r0, p0, alpha0 = self.point(psi), None, None, None
        v = lambda t: t[:, None, None, None]  # noqa: E731
        for n in range(iters):
            psi = pt["psi"]
            r = pt["H"] - v(pt["mu"]) * psi
            z = self.precondition(pt, r, mode)

            def direction(d):
                p = d - v(self.dot(d, psi)) * psi
                return p, float(self.dot(p, r).sum())

            beta = 0.0
            if n % 20:
                den = float(self.dot(r - r0, p0).sum())
                beta = max(float(self.dot(r - r0, z).sum()) / den, 0.0) if den else 0.0
            p, slope = direction(-z + beta * p0 if beta else -z)
            if slope >= 0.0 and beta:
                p, slope = direction(-z)
            if slope >= 0.0:
                p, slope = direction(-r)
            Ep, Epp = self.line(pt, p)
            pn = torch.sqrt(self.dot(p, p))
            model = Epp > 0.0
            alpha = -Ep / Epp if model else (alpha0 if alpha0 else math.pi / (4.0 * float(pn.max())))
            alpha = min(alpha, 0.5 * math.pi / float(pn.max()))
            for k in range(30):
                th = alpha * pn
                new = self.point(_unit(v(torch.cos(th)) * psi + v(torch.sin(th) / pn) * p, self.dV))
                if new["E"] < pt["E"] + tau * abs(pt["E"]) + (0.0 if model and k == 0 else 1e-4 * alpha * Ep):
                    break
                alpha *= 0.5
            pt, r0, p0, alpha0 = new, r, p, alpha
        return pt

    def ite(self, psi, dtau, steps):
        half = [torch.exp(-0.25 * dtau * self.k2)] * 2
        for _ in range(steps):
            psi = self.kin(psi, half)
            psi = self.kin(torch.exp(-dtau * self.point(psi)["U"]) * psi, half)
            psi = _unit(psi, self.dV)
        return self.point(psi)


def exact(case, seed):
    out = []
    for w, psi in _inputs(case, seed):
        m, op = _Plain(w), case["op"]
        psi = psi.to(torch.complex128)
        if op in ("energy_grad", "line_coeffs", "precondition", "autograd"):
            pt = m.point(psi)
            mu = [float(x) for x in pt["mu"]]
        if op == "energy_grad":
            return [pt["H"], pt["E"]] + mu
        if op == "line_coeffs":
            p = _direction(w, psi)
            p = p.to(torch.complex64).to(torch.complex128) if case["prec"] == "fp32" else p
            return [pt["E"], *m.line(pt, p)]
        if op == "precondition":
            r = pt["H"] - pt["mu"][:, None, None, None] * psi
            return [m.precondition(pt, r, case["precond"])]
        if op == "autograd":
            n, dV = pt["n"], m.dV
            Kn = [torch.fft.ifftn(m.kdd * torch.fft.fftn(n[i])).real for i in range(2)]
            _, F, d6 = m.lhy(n, eta=True)
            El, nt = float(dV * F.sum()), n[0] + n[1]
            s = lambda a, b: float(dV * (a * b).sum())  # noqa: E731
            d6 = [float(x) for x in d6]
            th = [0.5 * s(n[0], n[0]) + d6[0], s(n[0], n[1]) + d6[1], 0.5 * s(n[1], n[1]) + d6[2],
                  0.5 * s(n[0], Kn[0]) + d6[3], s(n[0], Kn[1]) + d6[4], 0.5 * s(n[1], Kn[1]) + d6[5],
                  El / w.kappa, -2.5 * El / w.eta_s]
            th += [w.trap[k] * float(dV * (q ** 2 * nt).sum()) for k, q in enumerate((m.x, m.y, m.z))]
            return [pt["E"], 2.0 * dV * pt["H"], torch.tensor(th, dtype=torch.float64)]
        if op == "ite":
            pt = m.ite(psi, case["dtau"], case["iters"])
        elif case["prec"] == "mixed":
            pt = m.ncg(psi, case["precond"], case["iters_fp32"], 1e-6)
            pt = m.ncg(pt["psi"], case["precond"], case["iters"], 1e-13)
        else:
            pt = m.ncg(psi, case["precond"], case["iters"], 1e-13 if case["prec"] == "fp64" else 1e-6)
        out.append([pt["psi"], pt["E"]] + [float(x) for x in pt["mu"]])
    return out

"""Performance cases: the runs a user of the library makes, through the C ABI's
binding (paper_1909_08390_gb300.fdlb), over the sizes of the repository's
workloads, tests and benchmark.

Kinds of cases:

* ``riemann``: an existing solver is set to two- or four-state Riemann data
  (fdlb_init_riemann), advanced ``steps`` IMEX steps, and its populations and
  moments are read into device arrays.  This is the loop of a parameter study
  or of a program that looks at the fields every ``steps`` steps.
* ``state``: the same from given populations (fdlb_set_state), periodic or
  outlet boxes: restarts, and programs that couple the solver to their own
  arrays.
* ``batch``: independent 1-D problems of uneven length in one context.
* ``grad``: the differentiable run (density_run): a loss of the final density
  and its gradient with respect to the initial fields and gamma.  (Not tau:
  it acts only through the populations' small distance from equilibrium, and
  at these tau that derivative carries rounding noise of about 1e-4.)

``exact`` is the method itself in plain torch, binary64: the literal stages of
the IMEX-SSP3(4,3,3) tableau, MP-9 with the Suresh-Huynh limiter, the
Gauss-Hermite moments and the Hermite-expanded equilibria.
"""
import math

import numpy as np
import torch

from paper_1909_08390_gb300 import fdlb, workloads as W

DEV = "cuda"
FP64, MIXED = fdlb.FDLB_FP64, fdlb.FDLB_MIXED


def listed():
    return [
        # One step and a look at the fields, 400-cell shock tube: the smallest
        # call, as in a coupled or interactive loop; launches and latency count.
        {"name": "tube400_one_step", "kind": "riemann", "d": 1, "nx": 400, "ny": 1, "qp": 8, "qc": 8,
         "prec": "fp64", "bc": 0, "steps": 1, "dt": 5e-5, "tau": 1e-6},
        # The shock tube of the paper's Fig. 1 at the step it keeps, the whole
        # run to t = 0.15 (300 steps of 5e-4 on 400 nodes, 8 populations).
        {"name": "tube400_fig1_run", "kind": "riemann", "d": 1, "nx": 400, "ny": 1, "qp": 5, "qc": 3,
         "prec": "fp64", "bc": 0, "steps": 300, "dt": 5e-4, "tau": 1e-5},
        # Fig. 1's finest grid with the full lattice in mixed precision; an odd
        # length.
        {"name": "tube3201_mixed", "kind": "riemann", "d": 1, "nx": 3201, "ny": 1, "qp": 8, "qc": 8,
         "prec": "mixed", "bc": 0, "steps": 128, "dt": 1e-5, "tau": 1e-5},
        # The benchmark problem (512 x 512, 8 x 8 velocities) in binary64.
        {"name": "quad512_fp64", "kind": "riemann", "d": 2, "nx": 512, "ny": 512, "qp": 8, "qc": 8,
         "prec": "fp64", "bc": 0, "steps": 4, "dt": 2.5e-5, "tau": 1e-6},
        # The same in mixed precision, one captured graph of steps.
        {"name": "quad512_mixed", "kind": "riemann", "d": 2, "nx": 512, "ny": 512, "qp": 8, "qc": 8,
         "prec": "mixed", "bc": 0, "steps": 16, "dt": 2.5e-5, "tau": 1e-6},
        # The paper's 2-D configuration size (400 x 400, Q = 5 and 3) in binary64.
        {"name": "lax400_fp64", "kind": "riemann", "d": 2, "nx": 400, "ny": 400, "qp": 5, "qc": 3,
         "prec": "fp64", "bc": 0, "steps": 16, "dt": 5e-4, "tau": 1e-5},
        # An odd and ragged 2-D grid in mixed precision (rows that are no
        # multiple of 4 cells).
        {"name": "ragged333x517_mixed", "kind": "riemann", "d": 2, "nx": 333, "ny": 517, "qp": 8,
         "qc": 8, "prec": "mixed", "bc": 0, "steps": 8, "dt": 2.5e-5, "tau": 1e-6},
        # The large problem: 2048 x 2048 cells, 128 populations, mixed precision.
        {"name": "quad2048_mixed", "kind": "riemann", "d": 2, "nx": 2048, "ny": 2048, "qp": 8,
         "qc": 8, "prec": "mixed", "bc": 0, "steps": 2, "dt": 2.5e-5, "tau": 1e-6},
        # A small periodic box from given populations, binary64, rectangular.
        {"name": "box96x70_periodic_fp64", "kind": "state", "d": 2, "nx": 96, "ny": 70, "qp": 8,
         "qc": 8, "prec": "fp64", "bc": 1, "steps": 16, "dt": 2e-4, "tau": 1e-5},
        # The 512-problem batch (lengths 256 to 4096, mixed precision).
        {"name": "batch512_mixed", "kind": "batch", "nprob": 512, "nlo": 256, "nhi": 4096, "qp": 8,
         "qc": 8, "prec": "mixed", "steps": 16, "dt": 2e-5, "tau": 1e-6},
        # A smaller batch with the paper's 1-D lattice in binary64.
        {"name": "batch96_fp64", "kind": "batch", "nprob": 96, "nlo": 256, "nhi": 4096, "qp": 5,
         "qc": 3, "prec": "fp64", "steps": 16, "dt": 2e-5, "tau": 1e-5},
        # Gradient of a density loss through 200 steps of the 2048-cell blended
        # tube, checkpoints every 50 steps.  The blend is wide enough that no
        # part of the domain is flat to rounding: there the limiter's choices,
        # and with them the gradient, would be decided by the last bit.
        {"name": "grad2048", "kind": "grad", "nx": 2048, "qp": 8, "qc": 8, "steps": 200, "every": 50,
         "dt": 5e-5, "tau": 1e-5, "width": 0.15},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _pmax(Q):
    return float(_nodes(Q)[0][-1])


def draw(rng):
    kind = rng.choice(["tube", "tube", "plane", "plane", "box", "batch", "grad"])
    qp, qc = rng.choice([(8, 8), (8, 8), (5, 3)])
    prec = rng.choice(["fp64", "mixed"])
    # |p| dt / dx as the workloads have it, 0.05 to 0.3
    cfl = rng.uniform(0.05, 0.3)
    tau = rng.choice([1e-6, 1e-5])
    if kind == "tube":
        nx = _log_int(rng, 100, 4096)
        return {"kind": "riemann", "d": 1, "nx": nx, "ny": 1, "qp": qp, "qc": qc, "prec": prec, "bc": 0,
                "steps": _log_int(rng, 1, 300), "dt": cfl / (nx * _pmax(qp)), "tau": tau}
    if kind == "plane":
        nx, ny = _log_int(rng, 40, 640), _log_int(rng, 40, 640)
        if rng.random() < 0.4:  # round sizes are common
            nx, ny = 16 * max(3, nx // 16), 16 * max(3, ny // 16)
        return {"kind": "riemann", "d": 2, "nx": nx, "ny": ny, "qp": qp, "qc": qc, "prec": prec,
                "bc": 0, "steps": rng.randint(2, 8), "dt": cfl / (max(nx, ny) * _pmax(qp)), "tau": tau}
    if kind == "box":
        d = rng.choice([1, 2])
        nx = _log_int(rng, 30, 3000 if d == 1 else 300)
        ny = 1 if d == 1 else _log_int(rng, 30, 300)
        return {"kind": "state", "d": d, "nx": nx, "ny": ny, "qp": qp, "qc": qc, "prec": prec,
                "bc": rng.choice([0, 1]), "steps": rng.randint(2, 20),
                "dt": cfl / (max(nx, ny) * _pmax(qp)), "tau": 1e-5}
    if kind == "batch":
        nlo = _log_int(rng, 64, 512)
        return {"kind": "batch", "nprob": _log_int(rng, 8, 512), "nlo": nlo,
                "nhi": _log_int(rng, 2 * nlo, 4096), "qp": qp, "qc": qc, "prec": prec,
                "steps": rng.randint(4, 20), "dt": 2e-5, "tau": tau}
    # to t = 0.01: the density feels gamma only at third order in t
    nx = _log_int(rng, 300, 1800)
    dt = rng.uniform(0.3, 0.45) / (nx * _pmax(qp))
    return {"kind": "grad", "nx": nx, "qp": qp, "qc": qc, "steps": math.ceil(0.01 / dt),
            "every": rng.choice([20, 25, 50]), "dt": dt, "tau": 1e-5, "width": rng.uniform(0.12, 0.2)}


# ---- inputs -------------------------------------------------------------------

def _domain(case):
    """[lo, hi] of both axes: the tubes' [-0.5, 0.5], the planes' [0, 1] (the
    paper's 2-D configurations, Q = 5 and 3, sit on [-0.5, 0.5])."""
    if case["d"] == 1 or case["qp"] == 5:
        return -0.5, 0.5
    return 0.0, 1.0


def _riemann_states(case, seed):
    """The workload's states, each value moved by up to 2 % by the seed."""
    base = ((W.SOD_LEFT, W.SOD_RIGHT) if case["d"] == 1 else
            W.C11_STATES if case["qp"] == 5 else W.quadrant_states(W.BENCH_SEED))
    rng = np.random.default_rng(seed)
    a = np.asarray(base, dtype=np.float64)
    return a * (1.0 + 0.02 * rng.uniform(-1.0, 1.0, a.shape))


def _populations(case, seed):
    """Positive populations away from equilibrium: the equilibrium of smooth
    periodic fields times a smooth factor within 2 %, made on the GPU."""
    d, nx, ny = case["d"], case["nx"], case["ny"]
    rng = np.random.default_rng(seed)
    x = (torch.arange(nx, dtype=torch.float64, device=DEV) + 0.5) / nx
    y = (torch.arange(ny, dtype=torch.float64, device=DEV) + 0.5) / ny

    def field(base, amp):
        f = torch.full((ny, nx), base, dtype=torch.float64, device=DEV)
        for mx in range(0, 3):
            for my in range(0, 3 if d == 2 else 1):
                if mx == my == 0:
                    continue
                c, ph = amp * rng.uniform(-1, 1) / (mx + my), rng.uniform(0, 2 * math.pi)
                f = f + c * torch.cos(2 * math.pi * (mx * x[None, :] + my * y[:, None]) + ph)
        return f

    fields = [field(1.0, 0.1), field(0.0, 0.1), field(0.0, 0.1) if d == 2 else None, field(1.0, 0.1)]
    if d == 1:
        fields = [None if f is None else f[0] for f in fields]
    m = _Model(d, case["qp"], case["qc"], 1.4)
    F = m.equilibrium(*fields)
    ph = torch.as_tensor(rng.uniform(0, 2 * math.pi, m.P), device=DEV)
    wave = 2 * math.pi * (x if d == 1 else x[None, :] + y[:, None])
    return F * (1.0 + 0.02 * torch.cos(wave[None] + ph.reshape((-1,) + (1,) * d)))


def _batch_inputs(case, seed):
    # lengths and gammas belong to the case, the gas states to the seed
    rng = np.random.default_rng(case["nprob"] + case["nlo"])
    nx = rng.integers(case["nlo"], case["nhi"] + 1, size=case["nprob"])
    gamma = rng.uniform(1.1, 5.0 / 3.0, size=case["nprob"])
    rng = np.random.default_rng(seed)
    st = np.empty((case["nprob"], 2, 3))
    st[:, :, 0] = rng.uniform(0.1, 1.0, (case["nprob"], 2))
    st[:, :, 1] = rng.uniform(-0.5, 0.5, (case["nprob"], 2))
    # temperatures P / rho of the range the lattice represents
    st[:, :, 2] = st[:, :, 0] * rng.uniform(0.6, 1.4, (case["nprob"], 2))
    return nx, gamma, st


def _grad_inputs(case, seed):
    rng = np.random.default_rng(seed)
    par = torch.as_tensor(np.asarray(W.SOD_LEFT + W.SOD_RIGHT) *
                          (1.0 + 0.02 * rng.uniform(-1, 1, 6)), dtype=torch.float64, device=DEV)
    fields = [f.contiguous() for f in fdlb.blended_fields(par, case["nx"], width=case["width"])]
    target = torch.as_tensor(W.smooth_target(case["nx"], seed=seed), device=DEV)
    return fields, target


def _precision(case):
    return FP64 if case["prec"] == "fp64" else MIXED


def prepare(case, seed):
    k = case["kind"]
    s = {"case": case}
    if k == "grad":
        fields, target = _grad_inputs(case, seed)
        one = lambda v: torch.tensor(v, dtype=torch.float64, device=DEV)
        s["inputs"] = [f.clone().requires_grad_(True) for f in fields + [one(1.4)]]
        s["tau"], s["target"] = one(case["tau"]), target
        s["spec"] = {"nx": case["nx"], "x0": -0.5, "x1": 0.5, "Q": (case["qp"], case["qc"]),
                     "dt": case["dt"], "nsteps": case["steps"], "every": case["every"]}
        return s
    if k == "batch":
        nx, gamma, st = _batch_inputs(case, seed)
        s["solver"] = fdlb.BatchSolver(nx, gamma, Qphi=case["qp"], Qchi=case["qc"], tau=case["tau"],
                                       dt=case["dt"], precision=_precision(case))
        s["states"] = st
    else:
        lo, hi = _domain(case)
        s["solver"] = fdlb.Solver(case["d"], case["nx"], case["ny"], lo, hi, lo, hi, case["bc"],
                                  case["qp"], case["qc"], 1.4, case["tau"], case["dt"],
                                  precision=_precision(case))
        if k == "state":
            s["F0"] = _populations(case, seed)
        else:
            s["states"] = _riemann_states(case, seed)
            s["split"] = 0.5 * (lo + hi)
    v = s["solver"]
    new = lambda *shape: torch.empty(shape, dtype=torch.float64, device=DEV)
    s["F"] = new(*v.shape)
    s["n"], s["ux"], s["T"] = (new(*v.shape[1:]) for _ in range(3))
    s["uy"] = new(*v.shape[1:]) if v.d == 2 else None
    return s


def run(s):
    case = s["case"]
    if case["kind"] == "grad":
        inputs = s["inputs"]
        n = fdlb.density_run(*inputs, s["tau"], s["spec"])
        loss = ((n - s["target"]) ** 2).sum() / case["nx"]
        return {"n": n.detach(), "loss": loss.detach(), "grads": torch.autograd.grad(loss, inputs)}
    v = s["solver"]
    if case["kind"] == "batch":
        v.init_riemann(s["states"])
        v.step(case["steps"], allow_unstable=True)
    else:
        if case["kind"] == "state":
            v.set_state(s["F0"])
        else:
            v.init_riemann(s["states"], s["split"], s["split"])
        v.step(case["steps"])
    fdlb.fdlb_get_state(v.ctx, s["F"], True)
    fdlb.fdlb_moments(v.ctx, s["n"], s["ux"], s["uy"], s["T"], True)
    return {"F": s["F"], "n": s["n"], "ux": s["ux"], "uy": s["uy"], "T": s["T"]}


def work(case):
    """Per step: the state read once and written once (8 bytes a population in
    either precision; a mixed state is a pair of binary32 values), and the
    operations of the three advected stages as bench.py counts them (an
    interface 24, two axes in 2-D, and each stage's update, moments and
    relaxation).  Then the state and the moments written out.  A gradient reads
    the forward's stages again and applies each one's transpose."""
    if case["kind"] == "batch":
        cells, d = int(_batch_inputs(case, 0)[0].sum()), 1
    else:
        d = case.get("d", 1)
        cells = case["nx"] * case.get("ny", 1)
    pops = case["qp"] ** d + case["qc"] ** d
    v = pops * cells
    flops = v * case["steps"] * (207 if d == 2 else 207 - 3 * 27)
    if case["kind"] == "grad":
        return {"bytes": 3 * 16 * v * case["steps"], "flops": 3 * flops}
    return {"bytes": 16 * v * case["steps"] + 8 * v + 8 * cells * (d + 2), "flops": flops}


# ---- the method in 64 bits -------------------------------------------------------

def _nodes(Q):
    x, w = np.polynomial.hermite_e.hermegauss(Q)
    return x, w / math.sqrt(2 * math.pi)


class _Model:
    """Lattice, moments and equilibria."""

    def __init__(self, d, qp, qc, gamma):
        self.d, self.qp, self.qc = d, qp, qc
        self.P = qp ** d + qc ** d
        self.nphi = qp ** d
        self.DK = 2.0 / (gamma - 1.0)
        self.kchi = self.DK - d
        px = np.concatenate([np.tile(_nodes(q)[0], q ** (d - 1)) for q in (qp, qc)])
        py = np.concatenate([np.repeat(_nodes(q)[0], q) if d == 2 else np.zeros(q) for q in (qp, qc)])
        self.p = (px, py)

    def axis(self, Q, u, T):
        """g_k = w_k sum_l He_l(p_k)/l! a_l(u, T), stacked over k."""
        x, w = _nodes(Q)
        a = [torch.ones_like(u), u]
        for l in range(2, Q):
            a.append(u * a[-1] + (l - 1) * (T - 1.0) * a[-2])
        he = [np.ones(Q), x]
        for l in range(2, Q):
            he.append(x * he[-1] - (l - 1) * he[-2])
        fact = [math.factorial(l) for l in range(Q)]
        return [sum(float(w[k] * he[l][k] / fact[l]) * a[l] for l in range(Q)) for k in range(Q)]

    def equilibrium(self, n, ux, uy, T):
        out = []
        for Q, s in ((self.qp, n), (self.qc, self.kchi * T * n)):
            gx = self.axis(Q, ux, T)
            if self.d == 1:
                out += [s * g for g in gx]
            else:
                out += [s * g * h for h in self.axis(Q, uy, T) for g in gx]
        return torch.stack(out)

    def moments(self, F):
        phi, chi = F[:self.nphi], F[self.nphi:]
        px, py = (torch.as_tensor(p[:self.nphi], device=F.device) for p in self.p)
        n = phi.sum(0)
        ux = torch.tensordot(px, phi, 1) / n
        uy = torch.tensordot(py, phi, 1) / n if self.d == 2 else None
        u2 = ux * ux + (uy * uy if self.d == 2 else 0.0)
        e = torch.tensordot(px * px + py * py, phi, 1) + chi.sum(0)
        return n, ux, uy, (e - n * u2) / (self.DK * n)

    def feq(self, F):
        return self.equilibrium(*self.moments(F))


def _least(a, b):
    return torch.where(a < b, a, b)


def _most(a, b):
    return torch.where(a < b, b, a)


def _minmod4(a, b):
    """minmod(4a - b, 4b - a, a, b); the first of equal magnitudes."""
    xs = (4 * a - b, 4 * b - a, a, b)
    same = ((xs[0] > 0) & (xs[1] > 0) & (a > 0) & (b > 0)) | ((xs[0] < 0) & (xs[1] < 0) & (a < 0) & (b < 0))
    r = xs[0]
    for x in xs[1:]:
        r = torch.where(x.abs() < r.abs(), x, r)
    return torch.where(same, r, torch.zeros_like(r))


_STENCIL = (-4, 37, -162, 479, 1120, -255, 50, -5)


def _face(v):
    """MP-9 interface value from the window v[0..8] = F_{s-4} .. F_{s+4}."""
    d = [v[k + 1] - v[k] for k in range(8)]
    a = sum(c * x for c, x in zip(_STENCIL, d)) / 2520
    cm, c0, c1 = d[3] - d[2], d[4] - d[3], d[5] - d[4]
    dmp, dmm = _minmod4(c0, c1), _minmod4(cm, c0)
    zero = torch.zeros_like(a)
    d0, md = d[4], 0.5 * (d[4] - dmp)
    ul, lc = 4 * d[3], 0.5 * d[3] + (4.0 / 3.0) * dmm
    lo = _most(_least(zero, _least(d0, md)), _least(zero, _least(ul, lc)))
    hi = _least(_most(zero, _most(d0, md)), _most(zero, _most(ul, lc)))
    return v[4] + _least(_most(a, lo), hi)


class _Grid:
    """Ghost-extended lines of one axis: `pad` lists the cell of each padded
    position, `left` the padded start of each cell's left interface window."""

    def __init__(self, lengths, bc, ds):
        pad, left, at = [], [], 0
        for n in lengths:
            i = np.arange(-5, n + 5)
            pad.append((i % n if bc else np.clip(i, 0, n - 1)) + (sum(lengths[:len(pad)]) if len(lengths) > 1 else 0))
            left.append(np.arange(n) + at)
            at += n + 10
        self.pad = torch.as_tensor(np.concatenate(pad), device=DEV)
        self.left = torch.as_tensor(np.concatenate(left), device=DEV)
        self.one = len(lengths) == 1
        self.ds = ds  # a number, or one per cell

    def gradient(self, F, p, axis):
        """p dF/ds along the axis for populations of one velocity sign (p >= 0
        marches the window upwards, p < 0 is the mirror image)."""
        G = F.index_select(axis, self.pad)
        up = p[0] >= 0
        n = G.shape[axis]
        f = _face([G.narrow(axis, m if up else 8 - m, n - 8) for m in range(9)])
        # p >= 0: the interface left of cell x starts at padded x; p < 0: at x + 1
        o = 0 if up else 1
        if self.one:
            m = n - 10
            df = f.narrow(axis, o + 1, m) - f.narrow(axis, o, m)
        else:
            df = f.index_select(axis, self.left + o + 1) - f.index_select(axis, self.left + o)
        pk = torch.as_tensor(p, device=F.device).reshape((-1,) + (1,) * (F.dim() - 1))
        return pk * df / self.ds


class _Imex:
    """The IMEX-SSP3(4,3,3) step, literally."""

    def __init__(self, model, grids, dt, tau):
        self.m, self.grids, self.dt, self.tau = model, grids, dt, tau
        al, be, et = 0.24169426078821, 0.06042356519705, 0.12915286960590
        self.At = [[0, 0, 0, 0], [0, 0, 0, 0], [0, 1, 0, 0], [0, 0.25, 0.25, 0]]
        self.A = [[al, 0, 0, 0], [-al, al, 0, 0], [0, 1 - al, al, 0], [be, et, 0.5 - be - et - al, al]]
        self.w = [0, 1 / 6, 1 / 6, 2 / 3]
        self.split = []
        for p in model.p[:model.d]:
            s = np.asarray(p) >= 0
            cut = [0] + [i for i in range(1, len(s)) if s[i] != s[i - 1]] + [len(s)]
            self.split.append([(a, min(a + 8, c)) for b, c in zip(cut, cut[1:]) for a in range(b, c, 8)])

    def advect(self, F):
        """dt p . grad F"""
        X = None
        for ax, (grid, blocks) in enumerate(zip(self.grids, self.split)):
            g = torch.cat([grid.gradient(F[a:b], self.m.p[ax][a:b], F.dim() - 1 - ax) for a, b in blocks])
            X = g if X is None else X + g
        return self.dt * X

    def step(self, F):
        lam = self.dt / self.tau
        X, dF = [], []
        for i in range(4):
            R = F
            for j in range(i):
                if self.At[i][j]:
                    R = R - self.At[i][j] * X[j]
                if self.A[i][j]:
                    R = R - self.A[i][j] * dF[j]
            dF.append(lam / (1 + self.A[i][i] * lam) * (R - self.m.feq(R)))
            X.append(self.advect(R - self.A[i][i] * dF[i]) if i else None)
        for i in range(1, 4):
            F = F - self.w[i] * (X[i] + dF[i])
        return F


def _sides(n, split_cells):
    return (np.arange(n) + 0.5 >= split_cells)


def _equilibrium_of(model, prim):
    """Populations of per-cell (rho, u.., P) arrays."""
    t = [torch.as_tensor(a, dtype=torch.float64, device=DEV) for a in prim]
    return model.equilibrium(t[0], t[1], t[2] if len(t) == 4 else None, t[-1] / t[0])


def exact(case, seed):
    k = case["kind"]
    if k == "grad":
        return _exact_grad(case, seed) if case["steps"] <= 240 else None
    with torch.no_grad():
        if k == "batch":
            nx, gamma, st = _batch_inputs(case, seed)
            prim = [np.concatenate([st[i, :, c][_sides(n, n / 2).astype(int)] for i, n in enumerate(nx)])
                    for c in range(3)]
            m = _Model(1, case["qp"], case["qc"], 1.4)
            m.DK = torch.as_tensor(np.repeat(2.0 / (gamma - 1.0), nx), device=DEV)
            m.kchi = m.DK - 1.0
            grids = [_Grid([int(n) for n in nx], 0, torch.as_tensor(np.repeat(1.0 / nx, nx), device=DEV))]
            F = _equilibrium_of(m, prim)
        else:
            d, nx, ny = case["d"], case["nx"], case["ny"]
            m = _Model(d, case["qp"], case["qc"], 1.4)
            grids = [_Grid([nx], case["bc"], 1.0 / nx)] + ([_Grid([ny], case["bc"], 1.0 / ny)] if d == 2 else [])
            if k == "state":
                F = _populations(case, seed)
            else:
                st = _riemann_states(case, seed)
                right = _sides(nx, nx / 2)
                if d == 1:
                    prim = [st[:, c][right.astype(int)] for c in range(3)]
                else:
                    up = _sides(ny, ny / 2)[:, None]
                    q = np.where(up, np.where(right, 0, 1), np.where(right, 3, 2))
                    prim = [st[:, c][q] for c in range(4)]
                F = _equilibrium_of(m, prim)
        f = _Imex(m, grids, case["dt"], case["tau"])
        for _ in range(case["steps"]):
            F = f.step(F)
        n, ux, uy, T = m.moments(F)
        return {"F": F, "n": n, "ux": ux, "uy": uy, "T": T}


def _exact_grad(case, seed):
    """Reverse mode through the same steps, one step's graph at a time; the
    selections of the limiter are constants of the derivative."""
    fields, target = _grad_inputs(case, seed)
    one = lambda v: torch.tensor(v, dtype=torch.float64, device=DEV)
    n0, u0, T0, gamma = [f.clone().requires_grad_(True) for f in fields + [one(1.4)]]

    def method(gamma):
        m = _Model(1, case["qp"], case["qc"], 1.4)
        m.DK = 2.0 / (gamma - 1.0)
        m.kchi = m.DK - 1.0
        return m, _Imex(m, [_Grid([case["nx"]], 0, 1.0 / case["nx"])], case["dt"], case["tau"])

    m, f = method(gamma)
    F0 = m.equilibrium(n0, u0, None, T0)
    kept = [F0.detach()]
    with torch.no_grad():
        for _ in range(case["steps"]):
            kept.append(f.step(kept[-1]))
    last = kept[-1].clone().requires_grad_(True)
    n = last[:m.nphi].sum(0)
    loss = ((n - target) ** 2).sum() / case["nx"]
    (bar,) = torch.autograd.grad(loss, last)
    dgamma = torch.zeros_like(gamma)
    for s in range(case["steps"] - 1, -1, -1):
        par, F = gamma.detach().requires_grad_(True), kept[s].requires_grad_(True)
        bar, dg = torch.autograd.grad((method(par)[1].step(F) * bar).sum(), [F, par])
        dgamma = dgamma + dg
    g = torch.autograd.grad((F0 * bar).sum(), [n0, u0, T0, gamma])
    return {"n": n.detach(), "loss": loss.detach(), "grads": [g[0], g[1], g[2], dgamma + g[3]]}

"""Performance cases of the time-domain Helmholtz preconditioner library.

Each case is work that a program using the library has it do through its public
entry points (``htd.Solver``, ``htd.Batch``, ``htd.htd_gmres_solve_host``):
applying the preconditioner, solving with FGMRES, running a batch, and
differentiating the recurrence.  Sizes, point densities, run lengths and layer
widths are those of the package's workloads, tests and benchmark, and sizes
between them; speeds and right-hand sides are drawn from the seed.

``exact`` restates the method (Stolk, arXiv 2006.16861: cell-form operator of
App. A, the integrators I_acd and I_abd, Table 1 and S_T read-outs, the
discrete adjoint) in 64-bit torch operations.
"""
from __future__ import annotations

import itertools
import math

import numpy as np
import torch

from paper_2006_16861_gb300 import htd, workloads


# ---- cases -------------------------------------------------------------------

def listed():
    return [
        # the smallest configuration in its plain FP64 form: a latency-bound
        # application, as inside a short solve
        dict(name="precond_2d_fp64_101", kind="precond", n="101x101", model="const", precision="fp64",
             mode="table1", ppw=10.0, layer=20),
        # an ordinary ragged 2-D grid with the complex-linear read-out S_T (two
        # real runs), the form the paper pairs with left GMRES
        dict(name="precond_2d_mixed_257x193_exact", kind="precond", n="257x193", model="grf",
             precision="mixed", mode="exact", ppw=8.0, layer=12),
        # the 2-D heterogeneous configuration: one application inside its solve
        dict(name="precond_2d_mixed_1001", kind="precond", n="1001x1001", model="grf",
             precision="mixed", mode="table1", ppw=8.0, layer=40),
        # a large, odd 2-D grid (beyond what the SMs' shared memory holds)
        dict(name="precond_2d_mixed_1501x2001", kind="precond", n="1501x2001", model="grf",
             precision="mixed", mode="table1", ppw=8.0, layer=40),
        # a large 2-D grid with the plain FP64 recurrence (reference solves)
        dict(name="precond_2d_fp64_801", kind="precond", n="801x801", model="grf", precision="fp64",
             mode="table1", ppw=8.0, layer=32),
        # the largest 3-D configuration: one application inside its solve
        dict(name="precond_3d_mixed_256", kind="precond", n="256x256x256", model="layered",
             precision="mixed", mode="table1", ppw=8.0, layer=24),
        # the shape of the paper's smallest 3-D example, at its 6 points per
        # wavelength and T = 25
        dict(name="precond_3d_mixed_106x200x200", kind="precond", n="106x200x200", model="layered",
             precision="mixed", mode="table1", ppw=6.0, layer=16, T=25),
        # 3-D with the plain FP64 recurrence (reference solves)
        dict(name="precond_3d_fp64_96", kind="precond", n="96x96x96", model="layered",
             precision="fp64", mode="table1", ppw=8.0, layer=9),
        # backward differences with non-diagonal (cell) damping
        dict(name="precond_2d_mixed_401_abd", kind="precond", n="401x401", model="grf",
             precision="mixed", mode="table1", ppw=8.0, layer=16, integrator="abd", damping="cell"),
        # a batch: a 3-D handle with several sources beside 2-D instances of
        # various sides, one application of every preconditioner
        dict(name="batch_mixed_64_8_plus_2d", kind="batch", n3=64, nrhs=8, sides="200,301,417,512,640",
             ppw=8.0),
        # a whole solve from host buffers to a true relative residual of 1e-6
        dict(name="solve_3d_mixed_128_host", kind="solve_host", n="128x128x128", model="layered",
             precision="mixed", ppw=8.0, layer=12),
        # the gradient of a receiver misfit through the recurrence (an inversion's
        # backward pass), several sources
        dict(name="grad_td_2d_mixed_512", kind="grad_td", n="512x512", model="grf", precision="mixed",
             ppw=8.0, layer=20, nsrc=4),
    ]


def draw(rng):
    def side(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["2d_mixed", "2d_mixed", "2d_fp64", "3d_mixed", "3d_mixed", "3d_fp64", "abd",
                       "batch", "grad_td"])
    mode = rng.choice(["table1", "table1", "exact", "project"])
    if kind in ("2d_mixed", "2d_fp64"):
        a = side(70, 1800 if kind == "2d_mixed" else 800)
        b = max(48, int(a * rng.uniform(0.6, 1.0)))
        if mode != "table1":
            a, b = min(a, 900), min(b, 900)
        n = rng.choice([(a, b), (b, a)])
        return dict(kind="precond", n="%dx%d" % n, model="grf", precision=kind[3:], mode=mode, ppw=8.0,
                    layer=max(6, int(0.04 * max(n))))
    if kind in ("3d_mixed", "3d_fp64"):
        a = side(32, 240 if kind == "3d_mixed" else 96)
        if mode != "table1":
            a = min(a, 150)
        n = [max(20, int(a * rng.uniform(0.5, 1.0))), max(20, int(a * rng.uniform(0.6, 1.0))), a]
        ppw = rng.choice([6.0, 8.0])
        return dict(kind="precond", n="%dx%dx%d" % tuple(n), model="layered", precision=kind[3:],
                    mode=mode, ppw=ppw, layer=max(3, int(round(24 * a / 256))))
    if kind == "abd":
        a = side(60, 700)
        if rng.random() < 0.5:
            n = "%dx%d" % (a, max(40, int(a * rng.uniform(0.6, 1.0))))
        else:
            a = min(a // 3, 128) + 20
            n = "%dx%dx%d" % (max(16, int(a * rng.uniform(0.6, 1.0))), a, max(16, a - rng.randint(0, 9)))
        return dict(kind="precond", n=n, model="grf" if n.count("x") == 1 else "layered",
                    precision=rng.choice(["mixed", "fp64"]) if a < 200 else "mixed", mode="table1",
                    ppw=8.0, layer=max(4, int(0.04 * a)), integrator="abd",
                    damping=rng.choice(["node", "cell"]))
    if kind == "batch":
        sides = ",".join(str(side(150, 800)) for _ in range(rng.randint(2, 6)))
        return dict(kind="batch", n3=side(32, 96), nrhs=rng.randint(1, 9), sides=sides, ppw=8.0)
    a = side(90, 512)
    return dict(kind="grad_td", n="%dx%d" % (a, max(64, int(a * rng.uniform(0.6, 1.0)))), model="grf",
                precision=rng.choice(["mixed", "mixed", "fp64"]), ppw=8.0,
                layer=max(6, int(0.04 * a)), nsrc=rng.randint(1, 4))


# ---- inputs (from the seed alone, made on the GPU) ----------------------------

def _sizes(case):
    return tuple(int(v) for v in case["n"].split("x"))


def _periods(case, n):
    """Periods per application: the longest side in wavelengths at the slowest speed."""
    return int(case.get("T") or max(1, math.ceil((max(n) - 1) / case["ppw"] - 1e-9)))


def _field(gen, shape, corr):
    """Zero-mean, unit-variance Gaussian random field with a Gaussian kernel of
    standard deviation `corr` cells (periodic)."""
    g = torch.randn(shape, generator=gen, device="cuda", dtype=torch.float64)
    f = torch.fft.rfftn(g)
    for ax, m in enumerate(shape):
        k = (torch.fft.rfftfreq(m, device="cuda", dtype=torch.float64) if ax == len(shape) - 1
             else torch.fft.fftfreq(m, device="cuda", dtype=torch.float64))
        view = [1] * len(shape)
        view[ax] = -1
        f = f * torch.exp(-2.0 * (math.pi * corr * k) ** 2).reshape(view)
    g = torch.fft.irfftn(f, s=shape)
    g = g - g.mean()
    return g / g.std()


def _model(n, model, ppw, layer, gen, damp=2.0):
    """Speed per cell, damping per node, h and omega: the package's three models
    (constant; 2-D random medium; 3-D layers with a random perturbation), with
    speeds of at least 1.5 (1 for the constant one) and omega set by it."""
    d, h = len(n), 1.0 / (max(n) - 1)
    cells = [m + 1 for m in n]
    cmin = 1.5
    if model == "const":
        c = torch.ones(cells, device="cuda", dtype=torch.float64)
        cmin = 1.0
    elif model == "grf":
        c = (3.0 + 0.75 * _field(gen, cells, 0.05 / h)).clamp(1.5, 4.5)
    else:
        depth = (torch.arange(cells[0], device="cuda", dtype=torch.float64) - 0.5) / (n[0] - 1)
        base = torch.tensor([1.5, 2.5, 3.5, 4.5], device="cuda", dtype=torch.float64)[
            (depth * 4).floor().clamp(0, 3).long()]
        c = base.reshape(-1, *[1] * (d - 1)) * (1.0 + 0.1 * _field(gen, cells, 0.05 / h))
        c = c.clamp(1.2, 5.5)
        cmin = 1.2
    omega = 2.0 * math.pi * cmin / (ppw * h)
    R = torch.zeros(n, device="cuda", dtype=torch.float64)
    for ax, m in enumerate(n):
        i = torch.arange(m, device="cuda", dtype=torch.float64)
        depth = (layer - torch.minimum(i, m - 1 - i)).clamp(min=0.0) / layer
        view = [1] * d
        view[ax] = -1
        R = R + damp * omega * (depth ** 2).reshape(view)
    return c, R, h, omega


def _dense(gen, shape):
    return torch.randn(shape, generator=gen, device="cuda", dtype=torch.complex128)


def _points(gen, n, h, nsrc, margin):
    """Point sources of amplitude 1/h^d at random nodes away from the layer."""
    F = torch.zeros((nsrc, *n), device="cuda", dtype=torch.complex128)
    for s in range(nsrc):
        pos = [margin + int(torch.randint(0, m - 2 * margin, (1,), generator=gen, device="cuda"))
               for m in n]
        F[(s, *pos)] = h ** -len(n)
    return F


def _inputs(case, seed):
    """Every system of the case as (n, c, R, h, omega, T, F)."""
    gen = torch.Generator(device="cuda").manual_seed(int(seed))
    if case["kind"] == "batch":
        n = (int(case["n3"]),) * 3
        layer = max(2, round(24 * n[0] / 256))
        sys = [(n, *_model(n, "layered", case["ppw"], layer, gen), _periods(case, n),
                _dense(gen, (case["nrhs"], *n)))]
        for side in (int(v) for v in case["sides"].split(",")):
            n = (side, side)
            sys.append((n, *_model(n, "grf", case["ppw"], max(4, round(0.04 * (side - 1))), gen),
                        _periods(case, n), _dense(gen, (1, *n))))
        return sys
    n = _sizes(case)
    # backward differences need weaker damping than the layer of the other cases
    damp = 0.25 if case.get("integrator") == "abd" else 2.0
    c, R, h, omega = _model(n, case["model"], case["ppw"], case["layer"], gen, damp)
    if case["kind"] == "precond":
        F = _dense(gen, n)                     # a Krylov vector: dense
    else:
        F = _points(gen, n, h, case.get("nsrc", 1), case["layer"] + 2)
        if case["kind"] == "solve_host":
            F = F[0]
    return [(n, c, R, h, omega, _periods(case, n), F)]


def _receivers(case):
    """Node indices on the first row inside the top layer, and their data's seed."""
    n, w = _sizes(case), case["layer"]
    return (w * n[1] + np.arange(w, n[1] - w)).astype(np.int64)


def _data(case, seed, h):
    gen = torch.Generator(device="cuda").manual_seed(int(seed) + 77)
    return _dense(gen, (case["nsrc"], _receivers(case).size))


def prepare(case, seed):
    probs = []
    for n, c, R, h, omega, T, F in _inputs(case, seed):
        probs.append((workloads.Problem("case", len(n), n, h, c.cpu().numpy(), R.cpu().numpy(), omega,
                                        None, T, 0.25), F))
    if case["kind"] == "batch":
        solvers = [htd.Solver(p, precision="mixed", max_rhs=int(F.shape[0])) for p, F in probs]
        batch = htd.Batch(solvers, [int(F.shape[0]) for _, F in probs])
        return dict(kind="batch", solvers=solvers, batch=batch, F=[F for _, F in probs],
                    U=batch.zeros())
    p, F = probs[0]
    opts = {k: case[k] for k in ("mode", "integrator", "damping") if k in case}
    s = htd.Solver(p, precision=case["precision"], **opts)
    state = dict(kind=case["kind"], solver=s, F=F)
    if case["kind"] == "precond":
        state["U"] = s.zeros()
    elif case["kind"] == "solve_host":
        state["F"] = F.cpu().pin_memory().numpy()
        state["U"] = torch.empty(F.shape, dtype=torch.complex128).pin_memory().numpy()
    else:
        state["rec"], state["d"] = _receivers(case), _data(case, seed, p.h)
    return state


def run(state):
    kind = state["kind"]
    if kind == "batch":
        return state["batch"].precond(state["F"], state["U"])
    s = state["solver"]
    if kind == "precond":
        return s.precond(state["F"], state["U"])
    if kind == "solve_host":
        state["U"].fill(0.0)
        info = htd.htd_gmres_solve_host(s.handle, state["F"], state["U"], 1e-6, 400)
        return dict(U=state["U"], iterations=info["iterations"])
    J, gm, gR = s.grad_td(state["F"], state["rec"], state["d"])
    return dict(J=J, grad_m=gm, grad_R=gR)


# ---- work ---------------------------------------------------------------------

# FLOPs of one point update: a multiply-add per stencil point and the update
def _update_flops(d):
    return 2.0 * 3 ** d + 8.0


def work(case):
    if case["kind"] == "batch":
        sys = [((case["n3"],) * 3, case["nrhs"])] + [((int(v),) * 2, 1) for v in case["sides"].split(",")]
    else:
        sys = [(_sizes(case), case.get("nsrc", 1))]
    flops = byts = 0.0
    for n, r in sys:
        N, d = math.prod(n), len(n)
        word = 8 if case.get("precision") == "fp64" else 4
        steps = _periods(case, n) * (8 if case["ppw"] <= 6.0 else 12)
        runs = {"exact": 2}.get(case.get("mode"), 1)
        if case["kind"] == "grad_td":
            # the application, then a forward and an adjoint run and one term per step
            flops += r * steps * N * (3 * _update_flops(d) + 2.0 * 4 ** d + 4.0)
            byts += r * N * 16 + N * (2 * word + 16)
        elif case["kind"] == "solve_host":
            # applications that a solve of this family takes
            flops += 30 * steps * N * _update_flops(d)
            byts += N * 32
        else:
            flops += r * runs * steps * N * _update_flops(d)
            byts += r * N * 32 + N * 2 * word
    return {"bytes": byts, "flops": flops}


# ---- 64-bit restatement ---------------------------------------------------------

class _Exact:
    """One system's operator, parameters and recurrence in 64-bit torch."""

    def __init__(self, n, c, R, h, omega, T, integrator="acd", damping="node"):
        self.n, self.d, self.h, self.w_phys, self.T = n, len(n), h, omega, T
        d = self.d
        third, sixth = 1.0 / 3.0, 1.0 / 6.0
        self.S, self.M = [], []
        for s in range(d + 1):
            q = 0.0
            if s > 0:
                q -= s * sixth ** (s - 1) * third ** (d - s)
            if s < d:
                q += (d - s) * sixth ** s * third ** (d - s - 1)
            self.S.append(q)
            self.M.append(0.5 * sixth ** s * third ** (d - s) + (0.5 ** (d + 1) if s == 0 else 0.0))
        kap = (h * omega / c) ** 2
        kmin, kmax = omega / float(c.max()), omega / float(c.min())
        # largest eigenvalue bound: the constant-coefficient symbol at k_min over {0, pi}^d
        k0 = (h * kmin) ** 2
        lam = -math.inf
        for v in itertools.product((1, -1), repeat=d):
            t = 0.0
            for o in itertools.product((-1, 0, 1), repeat=d):
                s = sum(abs(x) for x in o)
                t += 2.0 ** (d - s) * (self.S[s] - k0 * self.M[s]) * math.prod(
                    v[a] if o[a] else 1 for a in range(d))
            lam = max(lam, t)
        lam /= h * h
        w = kmax
        lam_im = omega * float(R.max())
        nP = 0
        while True:
            nP += 4
            th = 2 * math.pi / nP
            if integrator == "acd":
                if math.sin(math.pi / nP) ** 2 < w * w / (lam + w * w):
                    break
            else:
                al, be = th * th / (2 - 2 * math.cos(th)), th / math.sin(th)
                w2 = kmax * kmax + be / th * (1 - math.cos(th)) * lam_im
                if th * th / al * (lam / w2 + 1) + be / al * (1 + math.cos(th)) * lam_im / w2 < 4:
                    w = math.sqrt(w2)
                    break
        self.nP, self.w, self.N = nP, w, T * nP
        self.dt = 2 * math.pi / (w * nP)
        x = w * self.dt
        self.al, self.be = x * x / (2 - 2 * math.cos(x)), x / math.sin(x)
        self.cK = self.dt ** 2 / self.al
        self.integrator = integrator
        self.offs = list(itertools.product((-1, 0, 1), repeat=d))
        # (2 - K) per offset
        self.co = []
        for o, ks in zip(self.offs, self._shared(kap)):
            s = sum(abs(v) for v in o)
            wgt = (2.0 ** (d - s) * self.S[s] - self.M[s] * ks) / (h * h)
            wgt = -self.cK * wgt
            if s == 0:
                wgt = wgt + 2.0 - self.cK * w * w
            self.co.append(wgt)
        self.imH = omega * R
        ell = self.be * self.dt / self.al / w
        self.D = 1.0 / (1.0 + 0.5 * ell * self.imH)
        self.ell = ell
        self.ci = None
        if damping == "cell":
            pad = [1] * (2 * d)
            num = torch.nn.functional.pad(R, pad)
            one = torch.nn.functional.pad(torch.ones_like(R), pad)
            for ax in range(d):
                num = num.narrow(ax, 0, num.shape[ax] - 1) + num.narrow(ax, 1, num.shape[ax] - 1)
                one = one.narrow(ax, 0, one.shape[ax] - 1) + one.narrow(ax, 1, one.shape[ax] - 1)
            rc = omega * num / one
            self.ci = [self.M[sum(abs(v) for v in o)] * ks for o, ks in zip(self.offs, self._shared(rc))]

    def _shared(self, cell):
        """Sum of a cell array over the cells that a node shares with each neighbour."""
        for o in self.offs:
            v = cell
            for ax, k in enumerate(o):
                m = self.n[ax]
                lo, hi = v.narrow(ax, 0, m), v.narrow(ax, 1, m)
                v = lo if k < 0 else hi if k > 0 else lo + hi
            yield v

    def zeros(self):
        return torch.zeros([m + 2 for m in self.n], device="cuda", dtype=torch.float64)

    def inner(self, u, o=None):
        o = o or (0,) * self.d
        return u[tuple(slice(1 + k, 1 + k + m) for k, m in zip(o, self.n))]

    def apply(self, co, u):
        acc = co[0] * self.inner(u, self.offs[0])
        for w, o in zip(co[1:], self.offs[1:]):
            acc.addcmul_(w, self.inner(u, o))
        return acc

    def window(self, j, rho=0.25):
        s = 1.0 - j / self.N
        return 1.0 if s <= 1 - rho else math.sin(0.5 * math.pi * (1 - s) / rho) ** 2 if s < 1 else 0.0

    def step(self, u, um, g):
        """u_{j+1} into um (zero ring kept)."""
        t = self.apply(self.co, u)
        if g is not None:
            t += g
        p = self.inner(um)
        if self.integrator == "acd":
            p.copy_(self.D * (t - 2.0 * p) + p)
            return
        v = math.cos(2 * math.pi / self.nP) * u - um
        damp = self.apply(self.ci, v) if self.ci is not None else self.imH * self.inner(v)
        p.copy_(t - p - self.ell * damp)

    def force(self, j, fr, fi):
        ph = 2 * math.pi * (j % self.nP) / self.nP
        k = self.cK * self.window(j)
        return (k * math.cos(ph)) * fr - (k * math.sin(ph)) * fi

    def states(self, F):
        """Yields (j + 1, u_{j+1}) of the run with forcing F; the tensor is reused."""
        fr, fi = F.real.contiguous(), F.imag.contiguous()
        cur, oth = self.zeros(), self.zeros()
        for j in range(self.N):
            self.step(cur, oth, self.force(j, fr, fi))
            cur, oth = oth, cur
            yield j + 1, self.inner(cur)

    def precond(self, F, mode="table1"):
        if mode == "exact":
            for _, u in self.states(F):
                re = u
            re = re.clone()
            for _, u in self.states(-1j * F):
                im = u
            return torch.complex(re, im.clone())
        jim = self.N - self.nP // 4
        acc = torch.zeros(self.n, device="cuda", dtype=torch.complex128)
        for j, u in self.states(F):
            if mode == "project":
                if j > self.N - self.nP:
                    th = 2 * math.pi * (j % self.nP) / self.nP
                    acc += torch.complex(math.cos(th) * u, -math.sin(th) * u) * (2.0 / self.nP)
            elif j == jim:
                im = u.clone()
        return acc if mode == "project" else torch.complex(u.clone(), im)

    def grad_td(self, F, rec, data):
        J = 0.0
        gm = torch.zeros([m + 1 for m in self.n], device="cuda", dtype=torch.float64)
        gR = torch.zeros(self.n, device="cuda", dtype=torch.float64)
        jim = self.N - self.nP // 4
        corners = list(itertools.product((0, 1), repeat=self.d))

        def corner(u, b):
            return u[tuple(slice(k, k + m + 1) for k, m in zip(b, self.n))]

        for f, dd in zip(F, data):
            keep = [self.zeros(), self.zeros()]            # u_{-1}, u_0
            for j, u in self.states(f):
                s = self.zeros()
                self.inner(s).copy_(u)
                keep.append(s)                             # u_j at index j + 1
            res = torch.complex(self.inner(keep[self.N + 1]).reshape(-1)[rec],
                                self.inner(keep[jim + 1]).reshape(-1)[rec]) - dd
            J += 0.5 * float(res.abs().square().sum())
            are, aim = (torch.zeros(math.prod(self.n), device="cuda", dtype=torch.float64) for _ in "ab")
            are[rec] = res.real
            aim[rec] = res.imag
            la, lb = self.zeros(), self.zeros()
            for k in range(self.N, 0, -1):
                g = -are.reshape(self.n) if k == self.N else -aim.reshape(self.n) if k == jim else None
                self.step(la, lb, g)
                la, lb = lb, la
                # cell term, by sums over the corners' pairs
                u1 = keep[k]
                for b in corners:
                    t = None
                    for q in corners:
                        m = self.M[sum(x != y for x, y in zip(b, q))]
                        t = m * corner(u1, q) if t is None else t.add_(corner(u1, q), alpha=m)
                    gm.addcmul_(corner(la, b), t, value=-self.cK * self.w_phys ** 2)
                gR.addcmul_(self.inner(la), self.inner(keep[k + 1]) - self.inner(keep[k - 1]),
                            value=0.5 * self.ell * self.w_phys)
        return dict(J=J, grad_m=gm, grad_R=gR)


def exact(case, seed):
    if case["kind"] == "solve_host":
        return None                      # a 3-D direct solve takes too long
    out = []
    for n, c, R, h, omega, T, F in _inputs(case, seed):
        e = _Exact(n, c, R, h, omega, T, case.get("integrator", "acd"), case.get("damping", "node"))
        if case["kind"] == "grad_td":
            rec = torch.from_numpy(_receivers(case)).cuda()
            return e.grad_td(F, rec, _data(case, seed, h))
        if case["kind"] == "precond":
            return e.precond(F, case["mode"])
        out.append(torch.stack([e.precond(f) for f in F]))
    return out

"""The work this library is measured on: whole solves, gradients and single operators of the
all-at-once optimal-control system, each through the package's public entry points.

    listed()            the cases, dicts of plain values
    draw(rng)           one more case of the same ranges
    prepare(case, seed) the solver(s) and device inputs a program holds before the call
    run(state)          one pass
    work(case)          bytes and operations a pass cannot do without
    exact(case, seed)   what the pass returns, from plain torch in 64 bits

The FP32 and BF16-storage preconditioners are inner parts of flexible GMRES, so the mixed
cases are whole solves, which are defined by the system they solve; operators are measured
alone on FP64 handles and, where the entry point takes an FP32 vector, on that.  Solves return
the solution; the iteration count and residual that come with it describe the path to it.
"""
from __future__ import annotations

import math
from types import SimpleNamespace

import numpy as np
import torch

from paper_2410_22686_gb300 import Batch, Solver
from paper_2410_22686_gb300 import autograd as pcgrad

F64 = torch.float64


def _case(kind, dim, m1, n, **opt):
    """gamma: regularisation; eps: 'sqrt' sqrt(tau), 'half' 0.5 sqrt(tau), 'paper' min(1/2, tau/2);
    a: 'one', 'smooth' (2^s, s a smooth field in [-1, 1]) or 'field' (exp(0.5 G), G a Gaussian
    random field of correlation length 0.2); the rest are Solver / solve arguments."""
    c = dict(kind=kind, dim=dim, m1=m1, n=n, gamma=1e-4, eps="sqrt", a="smooth", space="fd", spatial="mg",
             precision="fp64", rtol=1e-8, mode="right", cap=60)
    c.update(opt)
    return c


def listed():
    return [
        # the smallest whole call: the plain configuration of the benchmark (61,504 unknowns), host-driven
        _case("solve", 2, 31, 32, name="solve_plain_31x32", gamma=1e-2, eps="half", a="one", spatial="fst"),
        # the paper's own experiments: n = 2^k - 1 time blocks, eps = tau/2, left-preconditioned GMRES
        _case("solve", 2, 63, 511, name="solve_paper_left_63x511", gamma=1e-2, eps="paper", a="one", spatial="fst",
              mode="left"),
        # the headline solve: variable coefficient, 33 M unknowns, FP32 preconditioner
        _case("solve", 2, 255, 256, name="solve_mixed_255x256", precision="fp32"),
        # the same discretisation solved in plain FP64 at an ordinary size
        _case("solve", 2, 127, 128, name="solve_fp64_127x128", gamma=1e-6),
        # the largest call: 3D random field, 64 M unknowns
        _case("solve", 3, 63, 128, name="solve_field_63c_128", a="field", precision="fp32"),
        # BF16-stored smoother iterates, an ordinary 2D size
        _case("solve", 2, 127, 64, name="solve_bf16s_127x64", gamma=1e-6, precision="bf16s"),
        # finite elements with a nodal coefficient in 2D and 3D
        _case("solve", 2, 127, 128, name="solve_fe_127x128", space="fe", precision="fp32", cap=80),
        _case("solve", 3, 31, 64, name="solve_fe_31c_64", a="field", space="fe", precision="fp32", cap=80),
        # many uneven problems in one graph launch (m1 x n of each)
        _case("batch", 2, 0, 0, name="batch_8_uneven", precision="fp32", cap=60,
              sizes="31x16 127x64 63x256 31x512 63x64 127x16 31x64 63x16"),
        # one training step of the coefficient and the target: forward, objective, adjoint, gradients
        _case("gradient", 2, 127, 128, name="gradient_127x128", rtol=1e-10, cap=80),
        # the preconditioner alone with odd sizes: neither the grid nor n is near a power of two
        _case("precond", 2, 100, 100, name="precond_odd_100x100", eps="paper", a="one", spatial="fst"),
        # the all-at-once product of the true residual, small enough that its latency counts
        _case("matvec", 2, 63, 64, name="matvec_63x64"),
    ]


def _logint(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["solve", "solve", "solve", "element", "left", "graph", "batch", "gradient", "precond", "matvec",
                       "matvec"])
    gamma = 10.0 ** rng.uniform(-8, -2)
    if kind == "batch":
        sizes = ["%dx%d" % (rng.choice([31, 63, 127]), rng.choice([16, 64, 256])) for _ in range(rng.randint(2, 8))]
        return _case("batch", 2, 0, 0, gamma=gamma, precision="fp32", sizes=" ".join(sizes))
    if kind == "left":
        # n = 2^k - 1 and the neighbouring lengths
        n = rng.choice([31, 63, 127, 255, 511, 1023]) - rng.choice([0, 0, 0, 1, 2])
        return _case("solve", 2, rng.choice([15, 31, 63]), n, gamma=10.0 ** rng.uniform(-4, -2), eps="paper", a="one",
                     spatial="fst", mode="left")
    if kind == "gradient":
        return _case("gradient", 2, rng.choice([31, 63, 127]), rng.choice([_logint(rng, 8, 128), 32, 64]),
                     gamma=10.0 ** rng.uniform(-5, -3), rtol=1e-10, cap=80)
    if kind == "element":
        dim = rng.choice([2, 3])
        m1 = rng.choice([31, 63, 127] if dim == 2 else [7, 15, 31])
        return _case("solve", dim, m1, 2 ** rng.randint(3, 7 if dim == 2 else 6), gamma=10.0 ** rng.uniform(-6, -3),
                     a="smooth" if dim == 2 else "field", space="fe", precision=rng.choice(["fp32", "fp64"]), cap=80)
    dim = rng.choice([2, 2, 3])
    const = rng.random() < 0.4
    if const:  # sine transforms take every m1
        m1 = _logint(rng, 9, 200) if dim == 2 else _logint(rng, 7, 40)
        more = dict(a="one", spatial="fst")
    else:
        m1 = rng.choice([31, 63, 127, 255] if dim == 2 else [7, 15, 31])
        more = dict(a="smooth" if dim == 2 else "field")
    room = 2.0e7 / m1 ** dim  # half vectors of at most 20 M values
    n = int(min(512, room, 2 ** rng.randint(3, 9)))
    if kind == "graph":
        n = 2 ** int(math.log2(max(2, min(n, 256))))
        return _case("graph", dim, m1, n, gamma=gamma, precision=rng.choice(["fp32", "fp64"]), **more)
    if rng.random() < 0.3:
        n = max(5, min(_logint(rng, 7, 300), int(room)))
    if kind == "solve":
        return _case("solve", dim, m1, n, gamma=gamma, precision=rng.choice(["fp32", "fp32", "fp64"]), **more)
    if kind == "precond":
        return _case("precond", dim, m1, n, gamma=gamma, eps=rng.choice(["sqrt", "half"]), **more)
    return _case(rng.choice(["matvec", "matvec_t", "matvec_f32"]), dim, m1, n, gamma=gamma,
                 space=rng.choice(["fd", "fd", "fe"]) if const else "fd", precision="fp32", **more)


# ------------------------------------------------------------------ inputs, from the seed alone

def _tau(c):
    return 1.0 / (c["n"] + 1)


def _eps(c):
    t = _tau(c)
    return {"sqrt": math.sqrt(t), "half": 0.5 * math.sqrt(t), "paper": min(0.5, 0.5 * t)}[c["eps"]]


def _coefficient(c, seed):
    """Nodal a, (m1+2)^dim, a numpy array; None for a = 1."""
    if c["a"] == "one":
        return None
    rng = np.random.default_rng(seed)
    m, d = c["m1"] + 2, c["dim"]
    if c["a"] == "smooth":
        x = np.linspace(0.0, 1.0, m)
        s = np.zeros((m, m))
        for _ in range(8):
            k = rng.integers(1, 4, size=2)
            ph = rng.uniform(0, 2 * math.pi, size=2)
            s += rng.standard_normal() * np.cos(math.pi * k[1] * x + ph[1])[:, None] * np.sin(math.pi * k[0] * x + ph[0])
        return 2.0 ** (s / np.abs(s).max())
    k = [2 * math.pi * np.fft.fftfreq(2 * m, d=1.0 / (m - 1))] * d
    k2 = sum(v ** 2 for v in np.meshgrid(*k, indexing="ij"))
    noise = np.fft.fftn(rng.standard_normal((2 * m,) * d))
    f = np.real(np.fft.ifftn(noise * np.exp(-0.01 * k2)))[(slice(0, m),) * d]
    return np.exp(0.5 * (f - f.mean()) / f.std())


def _target(c, seed):
    """g: 16 modes c sin(pi k1 x1) sin(pi k2 x2) .. cos(pi kt t), c ~ N(0, 1)."""
    rng = np.random.default_rng(seed + 77)
    d, m1, n = c["dim"], c["m1"], c["n"]
    x = torch.arange(1, m1 + 1, dtype=F64, device="cuda") / (m1 + 1)
    t = torch.arange(1, n + 1, dtype=F64, device="cuda") * _tau(c)
    ks, kt, amp = rng.integers(1, 5, size=(16, d)), rng.integers(0, 4, size=16), rng.standard_normal(16)
    g = torch.zeros((n,) + (m1,) * d, dtype=F64, device="cuda")
    for q in range(16):
        s = torch.ones((1,) * d, dtype=F64, device="cuda")
        for a in range(d):
            s = s * torch.sin(math.pi * int(ks[q, a]) * x).reshape([-1 if b == a else 1 for b in range(d)])
        g += float(amp[q]) * torch.cos(math.pi * int(kt[q]) * t).reshape((n,) + (1,) * d) * s
    return g


def _vector(c, seed, dtype=F64):
    gen = torch.Generator(device="cuda").manual_seed(seed)
    return torch.randn((2, c["n"]) + (c["m1"],) * c["dim"], dtype=dtype, device="cuda", generator=gen)


def _problems(c):
    """The single problems of a batch."""
    got = []
    for s in c["sizes"].split():
        m1, n = s.split("x")
        got.append(dict(c, kind="solve", m1=int(m1), n=int(n), gamma=c["gamma"] * 0.3 ** (len(got) % 4)))
    return got


def _solver(c, a):
    return Solver(c["dim"], c["m1"], c["n"], 1.0, c["gamma"], _eps(c), a, spatial=c["spatial"],
                  precision=c["precision"], max_iter=c["cap"], space=c["space"])


def prepare(case, seed):
    s = SimpleNamespace(c=case, kind=case["kind"])
    if s.kind == "batch":
        s.solvers, s.bs = [], []
        for k, c in enumerate(_problems(case)):
            s.solvers.append(_solver(c, _coefficient(c, seed + 1000 * k)))
            s.bs.append(s.solvers[-1].build_rhs(None, _target(c, seed + 1000 * k)))
        s.batch = Batch(s.solvers, s.bs, rtol=case["rtol"], maxit=case["cap"])
        return s
    a = _coefficient(case, seed)
    s.solver = _solver(case, a)
    if s.kind in ("solve", "graph"):
        s.b = s.solver.build_rhs(None, _target(case, seed))
        if s.kind == "graph":  # a graph is built for its buffers: the program keeps both
            s.x = torch.empty_like(s.b)
    elif s.kind == "gradient":
        s.log_a = torch.from_numpy(np.log(a[1:-1, 1:-1]).copy()).cuda()
        s.g = _target(case, seed)
    else:
        s.v = _vector(case, seed, torch.float32 if s.kind == "matvec_f32" else F64)
    return s


def run(s):
    c = s.c
    if s.kind == "solve":
        return s.solver.solve(s.b, rtol=c["rtol"], mode=c["mode"])[0]
    if s.kind == "graph":
        return s.solver.solve_graph(s.b, s.x, rtol=c["rtol"])[0]
    if s.kind == "batch":
        s.batch.solve()
        return s.batch.xs
    if s.kind == "gradient":
        la, g = s.log_a.clone().requires_grad_(True), s.g.clone().requires_grad_(True)
        J = pcgrad.objective(pcgrad.solve(s.solver, la, g, rtol=c["rtol"]), g, s.solver)
        J.backward()
        return {"J": J.detach(), "log_a": la.grad, "g": g.grad}
    if s.kind == "precond":
        return s.solver.apply_precond(s.v)
    if s.kind == "matvec_f32":
        return s.solver.matvec_f32(s.v)
    return s.solver.matvec(s.v, transpose=s.kind == "matvec_t")


# ------------------------------------------------------------------ what a pass cannot do without

def _iterations(c):
    """Iterations a solve takes, roughly: they grow with the digits asked for and with gamma."""
    at_1e8 = 16 if c["eps"] in ("paper", "half") else 25 + 2.2 * (8 + math.log10(c["gamma"]))
    return max(8, int(at_1e8 * -math.log10(c["rtol"]) / 8))


def _solve_work(c, iters):
    """Full GMRES: each iteration reads the basis (8 bytes a value) for the projections and again for
    the update, and applies preconditioner and operator once; the solution reads Z once."""
    u, zb = 2.0 * c["n"] * c["m1"] ** c["dim"], 4.0 if c["precision"] != "fp64" else 8.0
    fft = 5 * math.log2(max(2, c["n"])) + 40
    per = 16 * iters * (iters + 1) / 2 + iters * (24 + 2 * zb + zb + 8 + zb) + 24
    return {"bytes": u * per, "flops": u * (4 * iters * (iters + 1) / 2 + iters * (fft + 14))}


def work(case):
    if case["kind"] == "batch":
        w = [_solve_work(c, _iterations(c)) for c in _problems(case)]
        return {"bytes": sum(v["bytes"] for v in w), "flops": sum(v["flops"] for v in w)}
    u, d = 2.0 * case["n"] * case["m1"] ** case["dim"], case["dim"]
    if case["kind"] in ("solve", "graph"):
        return _solve_work(case, _iterations(case))
    if case["kind"] == "gradient":
        w = _solve_work(case, _iterations(case))
        return {"bytes": 2 * w["bytes"] + 80 * u, "flops": 2 * w["flops"] + 40 * u}
    if case["kind"] == "precond":
        side = 10 * d * math.log2(case["m1"] + 1) if case["spatial"] == "fst" else 40
        return {"bytes": 16 * u, "flops": u * (5 * math.log2(max(2, case["n"])) + side + 10)}
    nnz = 3 ** d if case["space"] == "fe" else 2 * d + 1
    return {"bytes": u * (12 if case["kind"] == "matvec_f32" else 16), "flops": u * (2 * nnz + 4)}


# ------------------------------------------------------------------ the same in plain torch, 64 bits

class _Plain:
    """M, K, T and A of one problem, written from the definitions: x = [half][time][space],
    A = [[alpha M, T^T], [-T, alpha M]], (T v)_j = M v_j - M v_{j-1} + tau K v_j."""

    def __init__(self, c, a):
        self.d, self.m, self.n, self.fe = c["dim"], c["m1"], c["n"], c["space"] == "fe"
        self.tau, self.h, self.N = _tau(c), 1.0 / (c["m1"] + 1), c["m1"] + 1
        self.gamma, self.alpha = c["gamma"], _tau(c) / math.sqrt(c["gamma"])
        self.a = torch.ones((self.m + 2,) * self.d, dtype=F64, device="cuda") if a is None else torch.from_numpy(a).cuda()
        th = math.pi * torch.arange(1, self.m + 1, dtype=F64, device="cuda") / self.N
        mean = float(torch.exp(torch.log(self.a).mean()))
        k1 = 4 * torch.sin(th / 2) ** 2 / (self.h if self.fe else self.h ** 2)
        m1 = self.h / 6 * (4 + 2 * torch.cos(th)) if self.fe else torch.ones_like(th)
        ax = lambda v, b: v.reshape([-1 if b == q else 1 for q in range(self.d)])  # noqa: E731
        self.mu = torch.ones((self.m,) * self.d, dtype=F64, device="cuda")
        self.lam = torch.zeros_like(self.mu)
        for b in range(self.d):
            self.mu = self.mu * ax(m1, b)
            part = torch.full_like(self.mu, mean)
            for q in range(self.d):
                part = part * ax(k1 if q == b else m1, q)
            self.lam = self.lam + part

    def sine(self, v):
        """The orthonormal DST-I along every space axis (its own inverse)."""
        for b in range(v.dim() - self.d, v.dim()):
            z = torch.zeros_like(v.narrow(b, 0, 1))
            f = torch.fft.rfft(torch.cat([z, v, z, -v.flip(b)], b), dim=b).imag.narrow(b, 1, self.m)
            v = f * (-0.5 * math.sqrt(2.0 / self.N))
        return v

    def mass(self, v):
        if not self.fe:
            return v
        for b in range(v.dim() - self.d, v.dim()):
            z = torch.zeros_like(v.narrow(b, 0, 1))
            p = torch.cat([z, v, z], b)
            v = (4 * v + p.narrow(b, 0, self.m) + p.narrow(b, 2, self.m)) * (self.h / 6)
        return v

    def mass_inv(self, v):
        return self.sine(self.sine(v) / self.mu) if self.fe else v

    def stiff(self, v, a=None):
        a = self.a if a is None else a
        lead = v.dim() - self.d
        if not self.fe:
            out, inner = 0, [slice(1, -1)] * self.d
            for b in range(self.d):
                lo, hi = list(inner), list(inner)
                lo[b], hi[b] = slice(0, -1), slice(1, None)
                face = 0.5 * (a[tuple(lo)] + a[tuple(hi)])
                z = torch.zeros_like(v.narrow(lead + b, 0, 1))
                out = out - (face * torch.cat([z, v, z], lead + b).diff(dim=lead + b)).diff(dim=lead + b)
            return out / self.h ** 2
        corners = list(np.ndindex(*(2,) * self.d))
        ae = sum(a[tuple(slice(i, i + self.N) for i in c)] for c in corners) / 2 ** self.d
        k1, m1 = np.array([[1, -1], [-1, 1]]) / self.h, np.array([[2, 1], [1, 2]]) * self.h / 6
        p = torch.nn.functional.pad(v, (1, 1) * self.d)
        out = torch.zeros_like(p)
        at = lambda t, c: t[(...,) + tuple(slice(i, i + self.N) for i in c)]  # noqa: E731
        for r in corners:
            acc = 0
            for q in corners:
                w = sum(math.prod((k1 if e == b else m1)[r[e], q[e]] for e in range(self.d)) for b in range(self.d))
                acc = acc + float(w) * at(p, q)
            at(out, r).add_(ae * acc)
        return out[(...,) + (slice(1, -1),) * self.d].contiguous()

    def T(self, v):
        mv = self.mass(v)
        out = mv + self.tau * self.stiff(v)
        out[1:] -= mv[:-1]
        return out

    def Tt(self, v):
        mv = self.mass(v)
        out = mv + self.tau * self.stiff(v)
        out[:-1] -= mv[1:]
        return out

    def A(self, x, sign=1.0):
        """A x, or A^T x with sign = -1."""
        return torch.stack([self.alpha * self.mass(x[0]) + sign * self.Tt(x[1]),
                            self.alpha * self.mass(x[1]) - sign * self.T(x[0])])

    def solve(self, b):
        """A^{-1} b: conjugate gradients on the Schur complement T (alpha M)^{-1} T^T + alpha M of p, preconditioned
        by (T_c + alpha M) (alpha M)^{-1} (T_c^T + alpha M) with the mean coefficient, refined on A itself."""
        al, den = self.alpha, self.mu * (1 + self.alpha) + self.tau * self.lam

        def pre(r):
            f = self.sine(r)
            f[0] /= den
            for j in range(1, self.n):
                f[j].addcmul_(self.mu, f[j - 1]).div_(den)
            f *= al * self.mu
            f[-1] /= den
            for j in range(self.n - 2, -1, -1):
                f[j].addcmul_(self.mu, f[j + 1]).div_(den)
            return self.sine(f)

        def schur(v):
            return self.T(self.mass_inv(self.Tt(v))) / al + al * self.mass(v)

        def once(r):
            rhs = r[1] + self.T(self.mass_inv(r[0])) / al
            x2, q = torch.zeros_like(rhs), rhs.clone()
            z = pre(q)
            p, rz = z, torch.sum(q * z)
            stop = 1e-12 * float(rz)
            for _ in range(200):
                sp = schur(p)
                step = rz / torch.sum(p * sp)
                x2 += step * p
                q -= step * sp
                z = pre(q)
                rz, old = torch.sum(q * z), rz
                if not float(rz) > stop:
                    break
                p = z + (rz / old) * p
            return torch.stack([self.mass_inv(r[0] - self.Tt(x2)) / al, x2])

        x, r, size = torch.zeros_like(b), b, float(b.norm())
        for _ in range(6):
            new = x + once(r)
            rn = b - self.A(new)
            if not float(rn.norm()) < float(r.norm()):
                break
            done = float(rn.norm()) > 0.3 * float(r.norm())
            x, r = new, rn
            if done or float(r.norm()) < 1e-16 * size:
                break
        return x

    def vcycle(self, s, r, a):
        """One V(1,0) cycle of (s I + tau K(a)): red-black Gauss-Seidel from zero, full weighting, linear prolongation."""
        m, d = r.shape[-1], self.d
        lev = SimpleNamespace(fe=False, d=d, h=1.0 / (m + 1), a=a)
        face = 0
        for b in range(d):
            e = [slice(1, -1)] * d
            lo, hi = list(e), list(e)
            lo[b], hi[b] = slice(0, -2), slice(2, None)
            face = face + 0.5 * (a[tuple(lo)] + 2 * a[tuple(e)] + a[tuple(hi)])
        dg = s + self.tau * face / lev.h ** 2
        if m == 1:
            return r / dg
        red = torch.from_numpy((np.indices((m,) * d).sum(0) + d) % 2 == 0).cuda()
        u = torch.where(red, r / dg, torch.zeros_like(r))
        off = s * u + self.tau * _Plain.stiff(lev, u) - dg * u
        u = torch.where(red, u, (r - off) / dg)
        res = r - s * u - self.tau * _Plain.stiff(lev, u)
        for b in range(1, d + 1):
            k = (m - 1) // 2
            at = lambda o: res.narrow(b, o, 2 * k - 1).index_select(b, torch.arange(0, 2 * k - 1, 2, device="cuda"))  # noqa: E731
            res = 0.5 * at(1) + 0.25 * (at(0) + at(2))
        e = self.vcycle(s, res, a[(slice(None, None, 2),) * d])
        for b in range(1, d + 1):
            z = torch.zeros_like(e.narrow(b, 0, 1))
            p = torch.cat([z, e, z], b)
            k = e.shape[b]
            mid = 0.5 * (p.narrow(b, 0, k + 1) + p.narrow(b, 1, k + 1))
            shape = list(e.shape)
            shape[b] = 2 * k + 1
            e = torch.stack([mid, torch.cat([e, z], b)], b + 1).flatten(b, b + 1).narrow(b, 0, 2 * k + 1).reshape(shape)
        return u + e

    def precond(self, v, eps, mg):
        n, col = self.n, (self.n,) + (1,) * self.d
        D = (eps ** (torch.arange(n, dtype=F64, device="cuda") / n)).reshape(col)
        th = 2 * math.pi * torch.arange(n, dtype=F64, device="cuda") / n
        sig = (1 - eps ** (1.0 / n) * torch.exp(-1j * th)).reshape(col) + self.alpha
        got = []
        for r, s in ((v[0] / D, sig.conj()), (v[1] * D, sig)):
            f = torch.fft.fft(r, dim=0)
            if mg:
                z = self.vcycle(s, f, self.a)
            else:
                t = torch.complex(self.sine(f.real), self.sine(f.imag)) / (s * self.mu + self.tau * self.lam)
                z = torch.complex(self.sine(t.real), self.sine(t.imag))
            got.append(torch.fft.ifft(z, dim=0).real)
        w1, w2 = got[0] * D, got[1] / D
        return torch.stack([w1 - w2, w1 + w2])


def _exact_solve(c, seed):
    p = _Plain(c, _coefficient(c, seed))
    b1 = p.tau * p.mass(_target(c, seed))
    return p.solve(torch.stack([b1, torch.zeros_like(b1)]))


def exact(case, seed):
    kind = case["kind"]
    if kind == "batch":
        return [_exact_solve(c, seed + 1000 * k) for k, c in enumerate(_problems(case))]
    if kind in ("solve", "graph"):
        return _exact_solve(case, seed)
    p = _Plain(case, _coefficient(case, seed))
    if kind == "gradient":
        g = _target(case, seed)
        b1 = p.tau * g
        x = p.solve(torch.stack([b1, torch.zeros_like(b1)]))
        y, w = x[0] / math.sqrt(p.gamma), p.h ** p.d * p.tau
        J = w * (0.5 * torch.sum((y - g) ** 2) + 0.5 / p.gamma * torch.sum(x[1] ** 2))
        dx = torch.stack([w * (y - g) / math.sqrt(p.gamma), w * x[1] / p.gamma])
        flip = torch.tensor([1.0, -1.0], dtype=F64, device="cuda").reshape((2,) + (1,) * (p.d + 1))
        lam = flip * p.solve(flip * dx)  # A^T = S A S, S = diag(I, -I)
        inner = (slice(1, -1),) * p.d
        la = torch.log(p.a[inner]).requires_grad_(True)
        a = p.a.clone()
        a[inner] = torch.exp(la)
        L = p.tau * (torch.sum(lam[0] * p.stiff(x[1], a)) - torch.sum(lam[1] * p.stiff(x[0], a)))
        return {"J": J, "log_a": -torch.autograd.grad(L, la)[0], "g": p.tau * lam[0] - w * (y - g)}
    s = _vector(case, seed, torch.float32 if kind == "matvec_f32" else F64).double()
    if kind == "precond":
        return p.precond(s, _eps(case), case["spatial"] == "mg")
    return p.A(s, -1.0 if kind == "matvec_t" else 1.0)

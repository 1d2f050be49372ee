"""The workloads that a user of this framework has it do, as measurable cases.

A case is one call (or one training step) through the package's public entry
points on a synthetic Gaia system of the paper's structure: rows grouped by
star and time-ordered inside a star, 5 astrometric + 12 attitude + 6
instrumental + 1 global nonzeros a row.  Values, true unknowns and noise are
drawn as in the package's generator (N(0, 1), N(0, 1), N(0, 1e-3)); a system's
shape is its number of stars, the mean number of observations a star
(Poisson, at least 10 of them; constant where "lam" is negative), the attitude
knots an axis and the instrument unknowns.

Tolerances are the entry points' own defaults (1e-12), at which a solve has
converged: its x is the least-squares solution, whatever the rounding.  The
standard errors follow the iteration count, and after many iterations the
rounding too, so solves ask for them where the observations of a star are
many (tens of iterations) and not where they are few.
"""
import math

import torch

from paper_2212_11675_gb300 import Solver, _lib, gen
from paper_2212_11675_gb300.autograd import GsrSolve

ITMAX = 2000      # of a PC-LSQR solve: never reached, the tolerances stop it
GRAD_TOL = 1e-13  # default tolerance of the adjoint's normal solve


def listed():
    return [
        # smallest calls: both products on the 1,000-star system, as an outer
        # method that keeps its own vectors calls them; launches and latency
        _case("products-1k", "products", 1000, -20, 200, 60),
        # y += A x and x += A^T y on the 100,000-star system (the benchmark's)
        _case("aprod1-100k", "aprod1", 100000, 70, 20000, 2000),
        _case("aprod2-100k", "aprod2", 100000, 70, 20000, 2000),
        # PC-LSQR on the 1,000-star system: many short iterations, as a
        # simulation campaign over small fields runs them
        _case("solve-1k", "solve", 1000, -20, 200, 60),
        # few stars with several hundred observations each (towards the
        # paper's thousand a star), all sizes odd
        _case("solve-deep", "solve", 2003, 400, 3001, 307),
        # the benchmark's system, solved to the default tolerance, with the
        # standard errors
        _case("solve-100k", "solve", 100000, 70, 20000, 2000),
        # a step towards the million-star systems, where the instrument
        # unknowns number several thousand
        _case("solve-wide", "solve", 170003, 70, 34001, 4001),
        # mixed precision: binary32 inner solve, FP64 refinement
        _case("mixed-10k", "mixed", 9973, 70, 1999, 211),
        _case("mixed-100k", "mixed", 100000, 70, 20000, 2000),
        # several right-hand sides at once: Monte Carlo noise realisations
        _case("batched8-100k", "batched", 100000, 70, 20000, 2000, 8),
        _case("batched19-10k", "batched", 10007, 61, 2003, 401, 19),
        # one training step of the differentiable solve: forward, backward
        # with respect to b and to the global column
        _case("gradient-20k", "gradient", 20000, 70, 4000, 400),
    ]


def _case(name, kind, stars, lam, knots, instr, k=1):
    return {"name": name, "kind": kind, "stars": stars, "lam": lam, "knots": knots,
            "instr": instr, "k": k, "se": kind == "solve" and lam >= 60}


def draw(rng):
    """Another call of the same ranges: 500 to 100,000 stars with 20 to 400
    observations each, attitude and instrument unknowns that they determine."""
    kind = rng.choice(("products", "aprod1", "aprod2", "solve", "solve", "mixed", "batched",
                       "gradient"))
    lam = int(round(math.exp(rng.uniform(math.log(20), math.log(400)))))
    top = min(100000, 7000000 // lam)
    k = 1
    if kind == "batched":
        k = rng.randint(2, 32)
        top = min(top, 24000000 // (k * lam))
    if kind == "gradient":
        top = min(top, 1400000 // lam)
    stars = int(round(math.exp(rng.uniform(math.log(500), math.log(top)))))
    rows = stars * lam
    knots = max(8, int(stars * math.exp(rng.uniform(math.log(0.1), math.log(0.4)))))
    instr = int(math.exp(rng.uniform(math.log(30), math.log(min(5000, max(60, rows // 300))))))
    c = _case("", kind, stars, lam, knots, instr, k)
    del c["name"]
    return c


# --------------------------------------------------------------------------
# inputs
# --------------------------------------------------------------------------
def _system(case, seed):
    """(star_ptr, attoff, instr, values, star of every row) on the GPU."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    # the survey's schedule (observations a star) belongs to the case
    gc = torch.Generator(device="cuda").manual_seed(case["stars"])
    S, D, I = case["stars"], case["knots"], case["instr"]
    f64 = dict(dtype=torch.float64, device="cuda")
    if case["lam"] < 0:
        cnt = torch.full((S,), -case["lam"], dtype=torch.int64, device="cuda")
    else:
        cnt = torch.poisson(torch.full((S,), float(case["lam"]), **f64), generator=gc)
        cnt = cnt.clamp(min=10).to(torch.int64)
    ptr = torch.zeros(S + 1, dtype=torch.int64, device="cuda")
    torch.cumsum(cnt, 0, out=ptr[1:])
    m = int(ptr[-1])
    star = torch.repeat_interleave(torch.arange(S, device="cuda"), cnt)
    # observation times, ascending inside each star
    t = (torch.sort(star + torch.rand(m, generator=g, **f64).clamp(max=0.999999))[0] - star)
    att = torch.floor(t.clamp(min=0.0) * (D - 3)).to(torch.int64).clamp(max=D - 4)
    # six distinct instrument unknowns a row (Floyd's sampling)
    ins = torch.empty((m, 6), dtype=torch.int64, device="cuda")
    u = torch.rand((m, 6), generator=g, **f64)
    for j in range(6):
        last = I - 6 + j
        v = (u[:, j] * (last + 1)).to(torch.int64).clamp(max=last)
        if j:
            v = torch.where((ins[:, :j] == v[:, None]).any(dim=1), torch.full_like(v, last), v)
        ins[:, j] = v
    values = torch.randn((m, 24), generator=g, **f64)
    return ptr, att, ins, values, star, g


def _cols(case, att, ins, star):
    """Column of each of the first 23 nonzeros of every row (the 24th is the
    last column), section by section."""
    S, D = case["stars"], case["knots"]
    j4 = torch.arange(4, device="cuda")
    yield slice(0, 5), 5 * star[:, None] + torch.arange(5, device="cuda")
    for a in range(3):
        yield slice(5 + 4 * a, 9 + 4 * a), 5 * S + a * D + att[:, None] + j4
    yield slice(17, 23), 5 * S + 3 * D + ins


class _Dense64:
    """A x and A^T y of a system in plain torch, 64 bits."""

    def __init__(self, case, sysm):
        _, att, ins, self.v, star, _ = sysm
        self.m, self.n = star.numel(), _n(case)
        self.parts = [(s, c) for s, c in _cols(case, att, ins, star)]

    def ax(self, x):
        y = self.v[:, 23] * x[-1]
        for s, c in self.parts:
            y = y + (self.v[:, s] * x[c]).sum(1)
        return y

    def aty(self, y):
        out = torch.zeros(self.n, dtype=torch.float64, device="cuda")
        for s, c in self.parts:
            out.index_add_(0, c.reshape(-1), (self.v[:, s] * y[:, None]).reshape(-1))
        out[-1] += (self.v[:, 23] * y).sum()
        return out

    def scale(self):
        """1 / column norms."""
        out = torch.zeros(self.n, dtype=torch.float64, device="cuda")
        for s, c in self.parts:
            out.index_add_(0, c.reshape(-1), self.v[:, s].square().reshape(-1))
        out[-1] += self.v[:, 23].square().sum()
        return torch.where(out > 0, out, torch.ones_like(out)).rsqrt()

    def normal(self, c, p, tol=1e-15, most=400):
        """(A^T A)^-1 c by conjugate gradients on the scaled columns."""
        s = p * c
        d, z = s.clone(), torch.zeros_like(s)
        gam = g0 = float(s @ s)
        for _ in range(most):
            if gam <= tol * tol * g0 or gam == 0.0:
                break
            q = self.ax(p * d)
            al = gam / float(q @ q)
            z += al * d
            s = s - al * (p * self.aty(q))
            new = float(s @ s)
            d = s + (new / gam) * d
            gam = new
        return p * z

    def solve(self, b, p):
        """argmin |A x - b|, refined twice on its own residual."""
        x = self.normal(self.aty(b), p)
        for _ in range(2):
            x = x + self.normal(self.aty(b - self.ax(x)), p, tol=1e-6)
        return x


def _n(case):
    return 5 * case["stars"] + 3 * case["knots"] + case["instr"] + 1


def _vectors(case, sysm):
    """The vectors of the call: a dict of tensors drawn after the system."""
    g, m, n = sysm[5], sysm[4].numel(), _n(case)

    def normal(*shape):
        return torch.randn(shape, generator=g, dtype=torch.float64, device="cuda")

    kind = case["kind"]
    if kind in ("products", "aprod1", "aprod2"):
        return {"x": normal(n), "y": normal(m), "y0": normal(m), "x0": normal(n)}
    x = normal(n)
    a = _Dense64(case, sysm)
    ax = a.ax(x)
    del a
    if kind == "batched":
        b = torch.empty((case["k"], m), dtype=torch.float64, device="cuda")
        for j in range(case["k"]):
            torch.add(ax, normal(m), alpha=1e-3, out=b[j])
        return {"b": b}
    v = {"b": ax + 1e-3 * normal(m)}
    if kind == "gradient":
        v["g"] = normal(n)  # gradient of the loss with respect to x
    return v


def prepare(case, seed):
    sysm = _system(case, seed)
    ptr, att, ins, values, _, _ = sysm
    state = {"kind": case["kind"], "se": case["se"], **_vectors(case, sysm)}
    system = gen.GaiaSystem(case["stars"], case["knots"], case["instr"], ptr.to(torch.uint32),
                            att.to(torch.uint32), ins.to(torch.uint16), values)
    torch.cuda.synchronize()  # gsr_create reads them on a stream of its own
    mixed = case["kind"] in ("mixed", "batched")
    state["solver"] = Solver(system,
                             precision=_lib.GSR_PREC_MIXED if mixed else _lib.GSR_PREC_FP64)
    if case["kind"] == "gradient":
        state["b"].requires_grad_(True)
        state["a"] = values[:, 23].contiguous().requires_grad_(True)
    return state


# --------------------------------------------------------------------------
# the calls
# --------------------------------------------------------------------------
def run(state):
    s, kind = state["solver"], state["kind"]
    if kind == "aprod1":
        return s.aprod1(state["x"], state["y0"])
    if kind == "aprod2":
        return s.aprod2(state["y"], state["x0"])
    if kind == "products":
        return {"y": s.aprod1(state["x"], state["y0"]), "x": s.aprod2(state["y"], state["x0"])}
    if kind == "solve":
        x, se, res = s.lsqr_solve(state["b"], ITMAX, want_se=state["se"])
        return {"x": x, "se": se, "rnorm": res["rnorm"], "istop": res["istop"]}
    if kind == "mixed":
        x, res = s.mixed_solve(state["b"])
        return {"x": x, "rnorm": res["rnorm"], "converged": res["converged"]}
    if kind == "batched":
        x, res = s.batched_solve(state["b"])
        return {"x": x, "rnorm": [r["rnorm"] for r in res],
                "converged": [r["converged"] for r in res]}
    b, a = state["b"], state["a"]
    b.grad = a.grad = None
    x = GsrSolve.apply(b, a, s, ITMAX)
    x.backward(state["g"])
    return {"x": x, "grad_b": b.grad, "grad_a": a.grad}


def exact(case, seed):
    sysm = _system(case, seed)
    v = _vectors(case, sysm)
    a = _Dense64(case, sysm)
    kind = case["kind"]
    if kind == "aprod1":
        return v["y0"] + a.ax(v["x"])
    if kind == "aprod2":
        return v["x0"] + a.aty(v["y"])
    if kind == "products":
        return {"y": v["y0"] + a.ax(v["x"]), "x": v["x0"] + a.aty(v["y"])}
    p = a.scale()
    if kind in ("solve", "mixed"):
        x = a.solve(v["b"], p)
        r = float((v["b"] - a.ax(x)).norm())
        return ({"x": x, "se": None, "rnorm": r, "istop": None} if kind == "solve" else
                {"x": x, "rnorm": r, "converged": None})
    if kind == "batched":
        b = v["b"]
        xs = torch.stack([a.solve(b[j], p) for j in range(b.shape[0])])
        return {"x": xs, "rnorm": [float((b[j] - a.ax(xs[j])).norm()) for j in range(len(b))],
                "converged": [None] * len(b)}
    x = a.solve(v["b"], p)
    q = a.normal(v["g"], p)
    q = q + a.normal(v["g"] - a.aty(a.ax(q)), p, tol=1e-6)
    sq, r = a.ax(q), v["b"] - a.ax(x)
    return {"x": x, "grad_b": sq, "grad_a": r * q[-1] - sq * x[-1]}


def _rows(case):
    return abs(case["lam"]) * case["stars"]


def _passes(case):
    """Passes over the matrix that a Krylov solve to 1e-12 takes: the residual
    falls by about (n / m)^0.32 a pass on these systems."""
    r = _n(case) / _rows(case)
    return math.ceil(math.log(1e12) / (0.32 * math.log(1.0 / r))) + 1


def work(case):
    """One pass over the matrix serves A x and A^T (A x): 24 values of 8 bytes
    and 16 bytes of indices a row, the m-vector read and written, n-vectors
    once a pass; the binary32 inner passes read 4-byte values."""
    m, n, k = _rows(case), _n(case), case["k"]
    kind = case["kind"]
    a64, a32 = 208.0 * m, 112.0 * m
    if kind in ("aprod1", "products"):
        w = {"bytes": a64 + 16.0 * m + 8.0 * n, "flops": 48.0 * m}
        if kind == "products":
            w = {"bytes": 2 * w["bytes"], "flops": 2 * w["flops"]}
        return w
    if kind == "aprod2":
        return {"bytes": a64 + 8.0 * m + 16.0 * n, "flops": 48.0 * m}
    its = _passes(case)
    if kind == "solve":
        return {"bytes": a64 + its * (a64 + 16.0 * m + 88.0 * n), "flops": its * (96.0 * m + 20 * n)}
    if kind == "gradient":
        return {"bytes": 2 * a64 + 2 * its * (a64 + 16.0 * m + 88.0 * n),
                "flops": 2 * its * (96.0 * m + 20 * n)}
    # the matrix is read once for all right-hand sides
    return {"bytes": a64 + its * (a32 + k * (8.0 * m + 64.0 * n)) + 4 * (a64 + k * 16.0 * m),
            "flops": (its + 4) * k * 96.0 * m}

"""Performance cases of the block-CG solver: what its users run, through the public entry points.

A user holds a gauge field (fat and long links) and a handle on it, and then
  * solves A X = B for a block of right-hand sides (BlockCG.solve; by far the most time),
    in the FP64-accurate form and in the mixed-precision forms;
  * applies the operator (apply_MdagM, dslash) to vectors of their own;
  * does block linear algebra on such blocks (block_cdot, block_caxpy, thin_qr);
  * differentiates a solve with respect to the links and the sources (hisq_solve);
  * solves many small independent problems together (BlockCGBatch).
Inputs are synthetic: links exp(0.3 i H) with Gaussian traceless Hermitian H (long links times
-1/24) and complex Gaussian sources, as in this repository's tests and benchmark.
"""
from __future__ import annotations

import math

import torch

LONG_COEFF = -1.0 / 24.0
EPS = 0.3
REAL_BYTES = {"f64": 8, "f64_native": 8, "mixed_f32": 4, "mixed_f16": 2, "mixed_bf16": 2}


# ------------------------------------------------------------------ the cases
def _case(name, kind, dims, n, mass, prec="f64", tol=1e-10, antiperiodic=False, seed_problems=0):
    lx, ly, lz, lt = dims
    c = {"kind": kind, "lx": lx, "ly": ly, "lz": lz, "lt": lt, "n": n, "mass": mass, "prec": prec,
         "tol": tol, "antiperiodic": antiperiodic}
    if kind == "batch":
        c["problems"], c["problem_seed"] = seed_problems
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # the smallest solve (smoke runs, unit tests, tiny lattices): launches and latency
        _case("solve-4^4-N4", "solve", (4, 4, 4, 4), 4, 0.1),
        # unequal extents, an odd block width, antiperiodic in time (the physical boundary condition)
        _case("solve-12.8.10.14-N5", "solve", (12, 8, 10, 14), 5, 0.05, antiperiodic=True),
        # the production solve: one block of 16 sources on a 32^4 lattice, FP64-accurate
        _case("solve-32^4-N16", "solve", (32, 32, 32, 32), 16, 0.01),
        # a wide block in the FP32 mixed form
        _case("solve-mixed32-24^4-N32", "solve", (24, 24, 24, 24), 32, 0.02, "mixed_f32"),
        # 16-bit storage with periodic reliable updates, to a tight residual
        _case("solve-mixed16-16^3x32-N16", "solve", (16, 16, 16, 32), 16, 0.05, "mixed_f16", tol=1e-12),
        # one source at a time, to a tight residual: the width-1 block many callers start from
        _case("solve-16^4-N1", "solve", (16, 16, 16, 16), 1, 0.05, tol=1e-12),
        # the operator on a production block, on the caller's layout
        _case("apply-32^4-N16", "apply", (32, 32, 32, 32), 16, 0.01),
        # the operator on a small lattice: a call inside somebody's own iteration
        _case("apply-8^4-N3", "apply", (8, 8, 8, 8), 3, 0.05),
        # one parity half on an odd width, at double precision throughout
        _case("dslash-native-16^3x24-N6", "dslash", (16, 16, 16, 24), 6, 0.05, "f64_native"),
        # block inner product, block update and thin QR on the caller's blocks
        _case("algebra-24^4-N12", "algebra", (24, 24, 24, 24), 12, 0.05),
        # forward and backward of a differentiable solve
        _case("grad-16^4-N8", "grad", (16, 16, 16, 16), 8, 0.05),
        # many small independent problems in one call (extents 8, 12 and 16, widths 2 to 16)
        _case("batch-24", "batch", (16, 16, 16, 16), 16, 0.01, "mixed_f32", seed_problems=(24, 4000)),
    ]


def draw(rng):
    """Another case of the same ranges: extents 4 to 32, widths 1 to 32, masses 0.01 to 0.2."""
    while True:
        kind = rng.choice(["solve", "solve", "solve", "solve", "apply", "dslash", "algebra", "grad", "batch"])
        dims = tuple(2 * round(math.exp(rng.uniform(math.log(2), math.log(16)))) for _ in range(4))
        n = min(32, int(math.exp(rng.uniform(0, math.log(33)))))
        mass = round(math.exp(rng.uniform(math.log(0.01), math.log(0.2))), 4)
        prec = rng.choice(["f64", "f64", "mixed_f32", "mixed_f16", "mixed_bf16", "f64_native"])
        anti = rng.random() < 0.5
        tol = 1e-12 if prec in ("mixed_f16", "mixed_bf16") else rng.choice([1e-11, 1e-12])
        rows = 3 * dims[0] * dims[1] * dims[2] * dims[3] // 2
        if kind == "batch":
            return _case(None, kind, (16, 16, 16, 16), 16, 0.01, "mixed_f32", 1e-10, False,
                         (rng.randint(4, 32), rng.randrange(1, 10000)))
        if kind in ("solve", "grad"):
            if kind == "grad":
                prec, tol = "f64", 1e-11
            # a block search space well below the vector space
            if rows / n < 2 * iterations(mass):
                continue
            if work_of_solve(dims, n, mass, prec) * (2 if kind == "grad" else 1) * (
                    8 if prec == "f64_native" else 1) > 0.7 * work_of_solve((32,) * 4, 16, 0.01, "f64"):
                continue
            if prec in ("mixed_f16", "mixed_bf16") and mass < 0.03:
                continue
        else:
            prec = rng.choice(["f64", "f64", "f64_native"])
            if rows / n < 8:
                continue
        return _case(None, kind, dims, n, mass, prec, tol, anti)


# ------------------------------------------------------------ inputs and plans
def _gell_mann(device):
    lam = torch.zeros((8, 3, 3), dtype=torch.complex128)
    for k, (i, j) in enumerate(((0, 1), (0, 2), (1, 2))):
        lam[2 * k, i, j] = lam[2 * k, j, i] = 1
        lam[2 * k + 1, i, j], lam[2 * k + 1, j, i] = -1j, 1j
    lam[6] = torch.diag(torch.tensor([1.0, -1.0, 0.0])).to(torch.complex128)
    lam[7] = torch.diag(torch.tensor([1.0, 1.0, -2.0])).to(torch.complex128) / math.sqrt(3)
    return lam.to(device)


def _exp_i(h, eps):
    """exp(i eps h) of traceless Hermitian 3x3 matrices: the power series in I, h and h^2, each power
    reduced with h^3 = (tr h^2 / 2) h + det h."""
    h2 = (h.unsqueeze(-1) * h.unsqueeze(-3)).sum(-2)
    c1 = h2.diagonal(dim1=-2, dim2=-1).sum(-1).real / 2
    c0 = (h2 * h.transpose(-1, -2)).sum((-2, -1)).real / 3
    a, b, c = torch.ones_like(c0), torch.zeros_like(c0), torch.zeros_like(c0)
    f, z = [torch.zeros_like(h[:, 0, 0]) for _ in range(3)], 1.0 + 0j
    for k in range(22):
        for fk, v in zip(f, (a, b, c)):
            fk += z * v
        z *= 1j * eps / (k + 1)
        a, b, c = c0 * c, a + c1 * c, b
    f0, f1, f2 = (v[:, None, None] for v in f)
    return f0 * torch.eye(3, dtype=h.dtype, device=h.device) + f1 * h + f2 * h2


def _links(dims, gen, device):
    """Fat exp(0.3 i H) and long -1/24 exp(0.3 i H') links, complex128 (4, V, 3, 3)."""
    v = dims[0] * dims[1] * dims[2] * dims[3]
    lam = (_gell_mann(device) / 2).reshape(8, 9)
    out = []
    for scale in (1.0, LONG_COEFF):
        u = torch.empty((4 * v, 3, 3), dtype=torch.complex128, device=device)
        for s in range(0, 4 * v, 1 << 20):
            e = min(4 * v, s + (1 << 20))
            w = torch.randn((e - s, 8), generator=gen, dtype=torch.float64, device=device)
            u[s:e] = _exp_i((w.to(torch.complex128) @ lam).reshape(-1, 3, 3), EPS) * scale
        out.append(u.view(4, v, 3, 3))
    return out


def _block(dims, n, gen, device):
    vh = dims[0] * dims[1] * dims[2] * dims[3] // 2
    return torch.complex(torch.randn((n, vh, 3), generator=gen, dtype=torch.float64, device=device),
                         torch.randn((n, vh, 3), generator=gen, dtype=torch.float64, device=device))


def _gen(seed, device):
    g = torch.Generator(device=device)
    g.manual_seed(int(seed) % (1 << 62))
    return g


def _dims(case):
    return (case["lx"], case["ly"], case["lz"], case["lt"])


def _batch_problems(case):
    """The shapes of the batch (not its fields): extents 8, 12 or 16, mass, width."""
    g = torch.Generator()
    g.manual_seed(case["problem_seed"])
    out = []
    for _ in range(case["problems"]):
        e = (8, 12, 16)[int(torch.randint(3, (1,), generator=g))]
        m = 0.01 + 0.19 * float(torch.rand((1,), generator=g))
        n = int(torch.randint(2, 17, (1,), generator=g))
        out.append(((e,) * 4, round(m, 4), n))
    return out


def _inputs(case, seed):
    dev = torch.device("cuda")
    gen = _gen(seed, dev)
    if case["kind"] == "batch":
        return [(d, m, n, *_links(d, gen, dev), _block(d, n, gen, dev))
                for d, m, n in _batch_problems(case)]
    d, n = _dims(case), case["n"]
    fat, lng = _links(d, gen, dev)
    x = _block(d, n, gen, dev)
    if case["kind"] == "algebra":
        a = torch.complex(torch.randn((n, n), generator=gen, dtype=torch.float64, device=dev),
                          torch.randn((n, n), generator=gen, dtype=torch.float64, device=dev))
        return fat, lng, x, _block(d, n, gen, dev), a
    return fat, lng, x


def prepare(case, seed):
    from paper_1710_09745_gb300 import BlockCG, BlockCGBatch

    if case["kind"] == "batch":
        solvers, blocks = [], []
        for d, m, n, fat, lng, b in _inputs(case, seed):
            solvers.append(BlockCG(d, fat, lng, m, prec=case["prec"], max_rhs=n))
            blocks.append(b)
        return {"case": case, "batch": BlockCGBatch(solvers), "blocks": blocks}
    fat, lng, *rest = _inputs(case, seed)
    s = BlockCG(_dims(case), fat, lng, case["mass"], prec=case["prec"], max_rhs=case["n"],
                antiperiodic_t=case["antiperiodic"])
    s.tune(case["n"])  # a program that keeps the handle tunes it once
    st = {"case": case, "solver": s, "rest": rest}
    if case["kind"] == "grad":
        st["leaves"] = [t.requires_grad_(True) for t in (fat, lng, rest[0])]
    return st


def run(state):
    case, kind = state["case"], state["case"]["kind"]
    if kind == "batch":
        xs, _, _ = state["batch"].solve(state["blocks"], tol=case["tol"])
        return xs
    s, rest = state["solver"], state["rest"]
    if kind == "solve":
        x, _ = s.solve(rest[0], tol=case["tol"])
        return x
    if kind == "apply":
        return s.apply_MdagM(rest[0])
    if kind == "dslash":
        return s.dslash(rest[0], out_parity=1)
    if kind == "algebra":
        x, y, a = rest
        q, r = s.thin_qr(x)
        return {"cdot": s.block_cdot(x, y), "caxpy": s.block_caxpy(x, a, y), "q": q, "r": r}
    from paper_1710_09745_gb300.autograd import hisq_solve

    fat, lng, phi = state["leaves"]
    for t in state["leaves"]:
        t.grad = None
    x = hisq_solve(fat, lng, phi, s, tol=case["tol"])
    loss = (phi.conj() * x).sum().real
    loss.backward()
    return {"loss": loss.detach(), "x": x.detach(), "fat": fat.grad, "lng": lng.grad, "phi": phi.grad}


# ------------------------------------------------------------------ the work
def iterations(mass):
    """Block-CG iterations to 1e-10 on these links, roughly (75 at m = 0.1, 270 at m = 0.01)."""
    return 27.0 / math.sqrt(mass)


def _per_iteration(dims, n, real):
    """(bytes, flops) of one iteration: two link sweeps, 14 passes over a block of n columns
    (the fused minimum), two stencil halves of 1158 flops per site and column, two Grams
    (one Hermitian product each) and four block products."""
    vh = dims[0] * dims[1] * dims[2] * dims[3] / 2
    return (2 * 288 * real * vh + 14 * 6 * n * real * vh,
            2 * 1158 * n * vh + (2 * 4 + 4 * 8) * n * n * 3 * vh)


def work_of_solve(dims, n, mass, prec):
    return iterations(mass) * _per_iteration(dims, n, REAL_BYTES[prec])[0]


def work(case):
    kind = case["kind"]
    if kind == "batch":
        w = [(d, n, m) for d, m, n in _batch_problems(case)]
        r = REAL_BYTES[case["prec"]]
        return {"bytes": sum(iterations(m) * _per_iteration(d, n, r)[0] for d, n, m in w),
                "flops": sum(iterations(m) * _per_iteration(d, n, r)[1] for d, n, m in w)}
    d, n = _dims(case), case["n"]
    vh = d[0] * d[1] * d[2] * d[3] // 2
    block, links = vh * n * 3 * 16, 2 * vh * 8 * 9 * 16
    if kind in ("solve", "grad"):
        b, f = _per_iteration(d, n, REAL_BYTES[case["prec"]])
        it = iterations(case["mass"])
        if kind == "solve":
            return {"bytes": it * b + 2 * block, "flops": it * f}
        # two solves, the links' gradients (an outer product per hop, both directions) and their output
        return {"bytes": 2 * it * b + 3 * block + 2 * links,
                "flops": 2 * it * f + 2 * 1158 * n * vh + 16 * 2 * 72 * n * vh}
    if kind in ("apply", "dslash"):
        halves = 2 if kind == "apply" else 1
        return {"bytes": 2 * block + links, "flops": halves * 1158.0 * n * vh}
    # K = X^H Y, Y + X a, X = Q R: each block read once per product, results written
    return {"bytes": 2 * block + 3 * block + 2 * block, "flops": (8 + 8 + 4 + 4) * 3.0 * vh * n * n}


# --------------------------------------------- 64-bit reference, plain torch
class _Reference:
    """The operator in complex128: fields (N, 3, Vh), links (3, 3, Vh) per parity and hop."""

    def __init__(self, dims, fat, lng, mass, antiperiodic):
        dev = fat.device
        lx, ly, lz, lt = dims
        self.m2 = mass * mass
        lex = torch.arange(lx * ly * lz * lt, device=dev)
        c = [lex % lx, lex // lx % ly, lex // (lx * ly) % lz, lex // (lx * ly * lz)]
        par = sum(c) % 2
        st = [1, lx, lx * ly, lx * ly * lz]
        self.hops = ([], [])
        for p in (0, 1):
            i = lex[par == p]
            ci = [x[i] for x in c]
            for mu in range(4):
                eta = 0.5 * (1 - 2 * (sum(ci[:mu]) % 2 if mu else torch.zeros_like(i))).to(torch.float64)
                for k, u in ((1, fat), (3, lng)):
                    for sgn in (1, -1):
                        w = ci[mu] + sgn * k
                        to = i + (w % dims[mu] - ci[mu]) * st[mu]
                        f = eta * sgn
                        if antiperiodic and mu == 3:
                            f = torch.where((w < 0) | (w >= lt), -f, f)
                        m = u[mu][i] if sgn > 0 else u[mu][to].mH
                        self.hops[p].append((to >> 1, (m * f[:, None, None]).permute(1, 2, 0)))

    def dslash(self, v, p):
        out = None
        for to, u in self.hops[p]:
            g = v[:, :, to]
            t = torch.stack([u[a, 0] * g[:, 0] + u[a, 1] * g[:, 1] + u[a, 2] * g[:, 2] for a in range(3)], 1)
            out = t if out is None else out + t
        return out

    def normal(self, v):
        return self.m2 * v - self.dslash(self.dslash(v, 1), 0)

    def solve(self, b, tol=3e-15, most=4000):
        """Conjugate gradients for all columns at once, restarted from the true residual."""
        n = b.shape[0]
        dot = lambda x, y: (x.conj() * y).real.reshape(n, -1).sum(1)  # noqa: E731
        bn = dot(b, b)
        x = torch.zeros_like(b)
        for restart in range(3):
            r = b - self.normal(x) if restart else b.clone()
            p, rr = r.clone(), dot(r, r)
            for it in range(most):
                ap = self.normal(p)
                al = rr / dot(p, ap).clamp_min(1e-300)
                x += al[:, None, None] * p
                r -= al[:, None, None] * ap
                new = dot(r, r)
                if it % 10 == 9 and float((new / bn).max()) < (tol if restart else 1e-12) ** 2:
                    break
                p = r + (new / rr.clamp_min(1e-300))[:, None, None] * p
                rr = new
        return x


def _to(v):
    return v.transpose(1, 2).contiguous()


def exact(case, seed):
    kind = case["kind"]
    if kind == "batch":
        out = []
        for k, (d, m, n, fat, lng, b) in enumerate(_inputs(case, seed)):
            out.append(_to(_Reference(d, fat, lng, m, False).solve(_to(b))) if k < 6 else None)
        return out
    d, n = _dims(case), case["n"]
    size = d[0] * d[1] * d[2] * d[3] * n * iterations(case["mass"])
    if kind in ("solve", "grad") and size > 24 ** 4 * 32 * iterations(0.02):
        return None  # over 20 seconds
    fat, lng, x, *more = _inputs(case, seed)
    if kind == "algebra":
        y, a = more
        xf, yf = x.reshape(n, -1), y.reshape(n, -1)
        low = torch.linalg.cholesky(xf.conj() @ xf.T)
        q = torch.linalg.solve_triangular(low.conj(), xf, upper=False)
        return {"cdot": xf.conj() @ yf.T, "caxpy": (yf + a.T @ xf).view_as(y), "q": q.view_as(x), "r": low.mH.resolve_conj()}
    if kind == "grad":
        r = _Reference(d, fat, lng, case["mass"], case["antiperiodic"])
        sol = r.solve(_to(x))
        # dL = -Re <lam, dA x> with lam = x for L = sum phi^H A^-1 phi
        y = r.dslash(sol, 1)
        leaves = [t.requires_grad_(True) for t in (fat, lng)]
        h = _Reference(d, *leaves, case["mass"], case["antiperiodic"])
        (2 * (sol.conj() * h.dslash(y, 0)).sum().real).backward()
        return {"loss": (_to(x).conj() * sol).sum().real, "x": _to(sol), "fat": leaves[0].grad,
                "lng": leaves[1].grad, "phi": 2 * _to(sol)}
    r = _Reference(d, fat, lng, case["mass"], case["antiperiodic"])
    v = _to(x)
    return _to(r.solve(v) if kind == "solve" else r.normal(v) if kind == "apply" else r.dslash(v, 1))

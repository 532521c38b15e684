"""The work that users of this package have it do, as cases of known size.

Each case names one call (or the few calls that belong together) of the public Python
binding, the mesh and options it runs on, and how its inputs are drawn:

  cycle   Context.vcycle: one multigrid cycle on a right-hand side, the preconditioner
          application that a user's own Krylov method makes (FP32 or FP64)
  stages  the steps a user composes a cycle of their own from: apply_agamma, star_smooth,
          restrict, prolong on the finest level
  solve   Context.update_coefficients + Context.solve: the step of a time loop or of a
          nonlinear iteration, setup for new coefficients and the solve with them
  batch   Batch.vcycle: the cycles of many small independent problems in one call

Inputs: multi-sinker viscosities (contrast `dr`) or, for `tensor`, the anisotropic
viscoplastic linearisation on top of them; right-hand sides are free of boundary values,
as residuals of a solve with Dirichlet data are.  `exact` restates the method densely in
64-bit torch, from element matrices, without this package's code.

FP32 cycles are taken with the P2 pairing, or with P1 at mild contrast, where a single
cycle is well conditioned with respect to rounding.
"""
import itertools
import math

import numpy as np
import torch

from paper_2107_00820_gb300 import Batch, Context
from paper_2107_00820_gb300 import alstokes as A

BATCH_MIX = "2d16x3,2d32x4,2d64x4,2d96x4,3d8x2,3d12x3,3d16x3,3d24x4"


def _case(name, kind, d, n, levels, **kw):
    n = (n,) * d if isinstance(n, int) else n
    c = {"name": name, "kind": kind, "d": d, "nx": n[0], "ny": n[1], "nz": n[2] if d == 3 else 1, "levels": levels,
         "order": 2, "prec": "fp32", "schur": "P2", "gamma": 10.0, "dr": 1e6, "sweeps": 5, "cycle": "V",
         "smoother": "gmres", "transfer": "robust", "tensor": False, "sinkers": 8 if d == 2 else 16}
    c.update(kw)
    return c


def listed():
    return [
        # the smallest calls: a two-level cycle on a mesh of a tutorial's size
        _case("cycle2d_16", "cycle", 2, 16, 2),
        # the 2D benchmark mesh, five levels
        _case("cycle2d_128", "cycle", 2, 128, 5, gamma=100.0),
        # a 2D channel in the default (FP64) mode, no power of two, P1 pairing at mild contrast
        _case("cycle2d_40x72_f64", "cycle", 2, (40, 72), 3, prec="fp64", schur="P1", dr=1e4),
        # the 3D benchmark mesh, four levels
        _case("cycle3d_32", "cycle", 3, 32, 4, dr=1e8),
        # a ragged 3D box, P1 pairing at mild contrast
        _case("cycle3d_20x28x12", "cycle", 3, (20, 28, 12), 3, schur="P1", dr=1e4),
        # 3D in the default (FP64) mode
        _case("cycle3d_16_f64", "cycle", 3, 16, 3, prec="fp64", gamma=100.0),
        # the higher-order element of the method's own runs, 2D and 3D
        _case("cycle2d_q3_128", "cycle", 2, 128, 5, order=3, gamma=100.0),
        _case("cycle3d_q3_12", "cycle", 3, 12, 3, order=3, gamma=1000.0),
        # the single steps on a ragged 3D level
        _case("stages3d_40x24x32", "stages", 3, (40, 24, 32), 3),
        # one step of a time loop: new coefficients, solve (the benchmark's workload)
        _case("solve3d_32", "solve", 3, 32, 4, prec="mixed", schur="P1", dr=1e6, rtol=1e-12),
        # one Newton step: anisotropic tensor coefficients
        _case("solve3d_tensor_16", "solve", 3, 16, 3, prec="mixed", tensor=True, gamma=1000.0, dr=1e6, rtol=1e-12),
        # a serving batch of uneven problems
        {"name": "batch_27", "kind": "batch", "mix": BATCH_MIX, "prec": "fp32", "schur": "P2", "gamma": 100.0,
         "dr": 1e6, "sweeps": 5},
    ]


def draw(rng):
    u = rng.random()
    if u < 0.1:
        # a batch of 4 to 24 problems
        mix = []
        for d, n in rng.sample([(2, 16), (2, 32), (2, 48), (2, 64), (2, 80), (3, 8), (3, 12), (3, 16), (3, 20)], 4):
            mix.append("%dd%dx%d" % (d, n, rng.randint(1, 6)))
        return {"kind": "batch", "mix": ",".join(mix), "prec": "fp32", "schur": "P2",
                "gamma": rng.choice([10.0, 100.0]), "dr": 10.0 ** rng.uniform(4, 8), "sweeps": rng.choice([3, 5])}
    kind = "cycle" if u < 0.7 else "stages" if u < 0.85 else "solve"
    d = rng.choice([2, 3])
    order = 3 if rng.random() < 0.2 and kind != "solve" else 2
    if d == 2:
        lo, hi = 12, {"solve": 64}.get(kind, 128 if order == 3 else 256)
    else:
        lo, hi = 6, {"solve": 16}.get(kind, 12 if order == 3 else 36)
    target = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    top = 10 if d == 2 else 5            # coarsest cells per axis: 4 .. 10 in 2D, 2 .. 5 in 3D
    levels = max(2, math.ceil(math.log2(target / top)) + 1)
    f = 2 ** (levels - 1)
    n = tuple(f * min(top, max(4 if d == 2 else 2, round(target * math.exp(rng.uniform(-0.3, 0.3)) / f)))
              for _ in range(d))
    p1 = rng.random() < 0.3
    prec = rng.choice(["mixed", "fp64"]) if kind == "solve" else "fp32" if rng.random() < 0.7 else "fp64"
    c = _case("", kind, d, n, levels, order=order, prec=prec, schur="P1" if p1 else "P2",
              gamma=rng.choice([10.0, 100.0]), dr=10.0 ** (rng.uniform(2, 4) if p1 else rng.uniform(4, 8)),
              sinkers=rng.randint(4, 24), tensor=order == 2 and not p1 and rng.random() < 0.15)
    if kind == "solve":
        c.update(rtol=1e-12, dr=min(c["dr"], 1e6), gamma=rng.choice([100.0, 1000.0]) if not p1 else c["gamma"])
    else:
        c.update(sweeps=rng.choice([2, 3, 5, 5, 5]), cycle="F" if rng.random() < 0.15 else "V",
                 smoother="richardson" if rng.random() < 0.12 else "gmres",
                 transfer="standard" if rng.random() < 0.08 else "robust")
    del c["name"]
    return c


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
def _sizes(c):
    n = (c["nx"], c["ny"], c["nz"])[: c["d"]]
    return [tuple(v // 2 ** (c["levels"] - 1 - l) for v in n) for l in range(c["levels"])]


def _grid(n, device):
    """Multi-indices of a box, first index fastest, (prod n, d)."""
    g = torch.meshgrid(*[torch.arange(v, device=device) for v in reversed(n)], indexing="ij")
    return torch.stack([t.reshape(-1) for t in reversed(g)], -1)


def _points(n, order, device):
    d = len(n)
    g = torch.tensor(np.polynomial.legendre.leggauss(order + 1)[0], device=device)
    q = g[_grid((order + 1,) * d, device)]
    h = torch.tensor([1.0 / v for v in n], dtype=torch.float64, device=device)
    return (_grid(n, device)[:, None, :] + 0.5 * (1.0 + q)[None]) * h


def _sinkers(x, centres, dr):
    """Viscosity of the multi-sinker law and its indicator 1 - chi."""
    d = x.shape[-1]
    chi = torch.ones(x.shape[:-1], dtype=torch.float64, device=x.device)
    for c in centres:
        s = (((x - c) ** 2).sum(-1).sqrt() - 0.5 * (0.1 if d == 2 else 0.15)).clamp(min=0.0)
        chi *= 1.0 - torch.exp(-200.0 * s * s)
    lo, hi = dr ** -0.5, dr ** 0.5
    return lo + (hi - lo) * (1.0 - chi), 1.0 - chi


def _tensor(x, mu, modes):
    """2 mu (I - alpha e e^T), e the unit Mandel strain of a smooth field, upper triangle."""
    m = 3 if x.shape[-1] == 2 else 6
    k, amp, ph = modes
    e = torch.cos(2 * math.pi * (x @ k.T) + ph) @ amp[:, :m]
    e = e / e.norm(dim=-1, keepdim=True).clamp(min=1e-12)
    alpha = 0.9 * (1.0 - mu / mu.max())
    C = 2.0 * mu[..., None, None] * (torch.eye(m, dtype=x.dtype, device=x.device)
                                     - alpha[..., None, None] * e[..., :, None] * e[..., None, :])
    iu = torch.triu_indices(m, m)
    return C[..., iu[0], iu[1]].contiguous()


def _problem(c, seed, device="cuda"):
    """Per-level coefficients (and mu_eff for tensors), force at the finest points."""
    g = torch.Generator().manual_seed(seed)
    d = c["d"]
    centres = torch.rand(c["sinkers"], d, generator=g, dtype=torch.float64).to(device)
    modes = (torch.randint(-3, 4, (8, d), generator=g).double().to(device),
             torch.randn(8, 6, generator=g, dtype=torch.float64).to(device),
             (2 * math.pi * torch.rand(8, generator=g, dtype=torch.float64)).to(device))
    coef, mu = [], []
    for n in _sizes(c):
        x = _points(n, c["order"], device)
        m, ind = _sinkers(x, centres, c["dr"])
        mu.append(m)
        coef.append(_tensor(x, m, modes) if c["tensor"] else m)
    f = torch.zeros(x.shape, dtype=torch.float64, device=device)
    f[..., -1] = -10.0 * ind
    return coef, mu if c["tensor"] else None, f


def _free(n, order, device):
    """Interior-node mask of the velocity lattice, per node."""
    nn = [order * v + 1 for v in n]
    ix = _grid(nn, device)
    top = torch.tensor(nn, device=device) - 1
    return ((ix > 0) & (ix < top)).all(-1)


def _vector(n, order, seed, dtype, device="cuda"):
    g = torch.Generator(device=device).manual_seed(seed)
    free = _free(n, order, device).repeat(len(n))
    return (torch.randn(free.numel(), generator=g, dtype=torch.float64, device=device) * free).to(dtype)


def _options(c):
    return {"mode": A.ALS_MODE_FP64 if c["prec"] == "fp64" else A.ALS_MODE_MIXED,
            "schur": A.ALS_SCHUR_P1 if c["schur"] == "P1" else A.ALS_SCHUR_P2,
            "sweeps": c["sweeps"],
            "smoother": A.ALS_SMOOTH_RICHARDSON if c.get("smoother") == "richardson" else A.ALS_SMOOTH_GMRES,
            "cycle": A.ALS_CYCLE_F if c.get("cycle") == "F" else A.ALS_CYCLE_V,
            "transfer": A.ALS_TRANSFER_STANDARD if c.get("transfer") == "standard" else A.ALS_TRANSFER_ROBUST,
            "order": c.get("order", 2)}


def _batch_cases(c):
    out = []
    for part in c["mix"].split(","):
        d, rest = int(part[0]), part[2:]
        n, count = (int(v) for v in rest.split("x"))
        floor, levels = 4 if d == 2 else 3, 1
        while n % 2 ** levels == 0 and n // 2 ** levels >= floor:
            levels += 1
        out += [_case("", "cycle", d, n, levels, schur=c["schur"], gamma=c["gamma"], dr=c["dr"], sweeps=c["sweeps"])
                for _ in range(count)]
    return out


def _dtype(c):
    return (torch.float32, A.ALS_PREC_FP32) if c["prec"] == "fp32" else (torch.float64, A.ALS_PREC_FP64)


def prepare(case, seed):
    c = case
    if c["kind"] == "batch":
        subs = _batch_cases(c)
        inst, b = [], []
        for i, s in enumerate(subs):
            coef, _, _ = _problem(s, 1000 * seed + i)
            inst.append({"dim": s["d"], "n": _sizes(s)[-1], "levels": s["levels"], "coeffs": coef,
                         "gamma": s["gamma"], "options": _options(dict(c, order=2))})
            b.append(_vector(_sizes(s)[-1], 2, 1000 * seed + i, torch.float32))
        return {"case": c, "batch": Batch(inst), "b": b, "x": [torch.zeros_like(t) for t in b]}
    coef, mu, f = _problem(c, seed)
    n = _sizes(c)[-1]
    opt = _options(c)
    if c["kind"] == "solve":
        opt.update(rtol=c["rtol"])
        coef0 = _problem(c, seed + 1)[0:2]      # the context is made for an earlier step's coefficients
        ctx = Context(c["d"], n, c["levels"], coef0[0], c["gamma"], mu_eff=coef0[1], **opt)
        z = {"u": torch.zeros(ctx.nu(), dtype=torch.float64, device="cuda"),
             "p": torch.zeros(ctx.npres(), dtype=torch.float64, device="cuda")}
        return {"case": c, "ctx": ctx, "coef": coef, "mu": mu, "f": f, **z}
    ctx = Context(c["d"], n, c["levels"], coef, c["gamma"], mu_eff=mu, **opt)
    dt, _ = _dtype(c)
    b = _vector(n, c["order"], seed, dt)
    s = {"case": c, "ctx": ctx, "b": b, "x": torch.zeros_like(b)}
    if c["kind"] == "stages":
        s["c"] = _vector(_sizes(c)[-2], c["order"], seed + 1, dt)
        s.update(y=torch.zeros_like(b), rc=torch.zeros_like(s["c"]), xf=torch.zeros_like(b))
    return s


def run(state):
    c = state["case"]
    if c["kind"] == "batch":
        state["batch"].vcycle(state["b"], state["x"], prec=A.ALS_PREC_FP32)
        return state["x"]
    ctx = state["ctx"]
    if c["kind"] == "solve":
        ctx.update_coefficients(state["coef"], state["mu"])
        u, p, _ = ctx.solve(state["f"], u=state["u"], p=state["p"])
        return {"u": u, "p": p}
    prec = _dtype(c)[1]
    if c["kind"] == "cycle":
        ctx.vcycle(state["b"], state["x"], prec=prec)
        return state["x"]
    top = c["levels"] - 1
    ctx.apply_agamma(state["b"], state["y"], prec=prec)
    ctx.star_smooth(top, state["b"], state["x"], prec=prec)
    ctx.restrict(top, state["b"], state["rc"], prec=prec)
    ctx.prolong(top, state["c"], state["xf"], prec=prec)
    return {"Ab": state["y"], "Db": state["x"], "restricted": state["rc"], "prolonged": state["xf"]}


# ---------------------------------------------------------------------------
# work
# ---------------------------------------------------------------------------
def _level_work(c, n, es):
    """(bytes, flops) of one operator apply and of one sweep of star products on a level.

    Apply: x, y, the coefficients; star sweep: the packed symmetric inverses, r, z.  The
    inverses of a sweep are counted at every sweep: the next one needs this one's result
    everywhere, and those of the large levels do not fit on the chip."""
    d, k = c["d"], c.get("order", 2)
    cells, verts = math.prod(n), math.prod(v - 1 for v in n)
    nu = d * math.prod(k * v + 1 for v in n)
    q = k + 1
    ncoef = (6 if d == 2 else 21) if c.get("tensor") else 1
    npd = d * (2 * k - 1) ** d
    stages = 2 * (d * (d + 1) // 2 + 1) * d        # 1D contractions of one sum-factorised apply
    apply_ = (2 * nu * es + cells * q ** d * ncoef * es, cells * q ** d * (stages * 2 * q + 30 + 4 * ncoef))
    star = (2 * nu * es + verts * npd * (npd + 1) // 2 * es, verts * 2 * npd * npd)
    return apply_, star


def _cycle_work(c, es):
    b = f = 0.0
    sizes = _sizes(c)
    visits = 1
    for l in range(len(sizes) - 1, 0, -1):
        (ab, af), (sb, sf) = _level_work(c, sizes[l], es)
        s = c["sweeps"]
        robust = 1 if c.get("transfer", "robust") == "robust" else 0
        b += visits * ((2 * s + 1 + 2 * robust) * ab + (2 * s + robust / 2 ** (c["d"] - 1)) * sb)
        f += visits * ((2 * s + 1 + 2 * robust) * af + (2 * s + robust / 2 ** (c["d"] - 1)) * sf)
        if c.get("cycle") == "F" and l > 1:
            visits += 1
    m = c["d"] * math.prod(c.get("order", 2) * v - 1 for v in sizes[0])
    return b + visits * 4.0 * m * m, f + visits * 2.0 * m * m


def work(case):
    c = case
    if c["kind"] == "batch":
        ws = [_cycle_work(s, 4) for s in _batch_cases(c)]
        return {"bytes": sum(w[0] for w in ws), "flops": sum(w[1] for w in ws)}
    es = 8 if c["prec"] == "fp64" else 4
    if c["kind"] == "cycle":
        b, f = _cycle_work(c, es)
        return {"bytes": b, "flops": f}
    if c["kind"] == "stages":
        (ab, af), (sb, sf) = _level_work(c, _sizes(c)[-1], es)
        part = 2.0 / 2 ** c["d"]          # the transfers' local solves: one star in 2^d, twice
        return {"bytes": 3 * ab + (1 + part) * sb, "flops": 3 * af + (1 + part) * sf}
    # solve: the stars' elimination, and about 40 iterations of two cycles and one FP64 apply
    b, f = _cycle_work(c, es)
    (ab, af), (sb, _) = _level_work(c, _sizes(c)[-1], 8)
    npd = c["d"] * 3 ** c["d"]
    verts = sum(math.prod(v - 1 for v in n) for n in _sizes(c)[1:])
    return {"bytes": 80 * b + 40 * ab + sb, "flops": 80 * f + 40 * af + verts * float(npd) ** 3}


# ---------------------------------------------------------------------------
# exact: the method from dense element and star matrices, 64 bits
# ---------------------------------------------------------------------------
class _Ref:
    """One level: element matrices, constrained operator, stars."""

    def __init__(self, c, n, coef, mu, stars=True):
        dev = coef.device
        d, k = len(n), c.get("order", 2)
        self.d, self.k, self.n = d, k, n
        g, w = np.polynomial.legendre.leggauss(k + 1)
        t = np.linspace(-1.0, 1.0, k + 1)
        basis = [np.polynomial.Polynomial.fromroots(np.delete(t, a)) for a in range(k + 1)]
        basis = [p / p(t[a]) for a, p in enumerate(basis)]
        L = np.array([[p(x) for p in basis] for x in g])
        D = np.array([[p.deriv()(x) for p in basis] for x in g])
        mi = np.array(list(itertools.product(range(k + 1), repeat=d)))[:, ::-1]
        nb = len(mi)
        wdet = np.prod(w[mi], axis=1) * np.prod([0.5 / v for v in n])
        grad = np.ones((nb, nb, d))
        for j in range(d):
            for a in range(d):
                grad[:, :, j] *= (D if a == j else L)[mi[:, a][:, None], mi[:, a][None, :]]
            grad[:, :, j] *= 2.0 * n[j]
        exps = [e for e in itertools.product(range(k), repeat=d) if sum(e) < k]
        exps.sort(key=lambda e: (sum(e), [-v for v in e]))
        psi = np.stack([np.prod(g[mi] ** np.array(e), axis=1) for e in exps], -1)
        self.npr, self.psi, self.wdet, self.phi = psi.shape[1], psi, wdet, np.ones((nb, nb))
        for a in range(d):
            self.phi *= L[mi[:, a][:, None], mi[:, a][None, :]]
        m = d * nb
        eps = np.zeros((nb, m, d, d))
        for a in range(d):
            eps[:, a * nb:(a + 1) * nb, a, :] += 0.5 * grad
            eps[:, a * nb:(a + 1) * nb, :, a] += 0.5 * grad
        div = np.concatenate([grad[:, :, a] for a in range(d)], axis=1)
        tt = lambda v: torch.as_tensor(np.ascontiguousarray(v), dtype=torch.float64, device=dev)  # noqa: E731
        if c.get("tensor"):
            prs = [(0, 0), (1, 1), (0, 1)] if d == 2 else [(0, 0), (1, 1), (2, 2), (1, 2), (0, 2), (0, 1)]
            mv = tt(np.stack([eps[:, :, i, j] * (1.0 if i == j else math.sqrt(2.0)) for i, j in prs], -1))
            nm = len(prs)
            iu = torch.triu_indices(nm, nm)
            C = torch.zeros(coef.shape[:2] + (nm, nm), dtype=torch.float64, device=dev)
            C[..., iu[0], iu[1]] = coef
            C[..., iu[1], iu[0]] = coef
            K = sum(wdet[q] * (mv[q] @ C[:, q] @ mv[q].T) for q in range(nb))
        else:
            T = np.einsum("q,qikl,qjkl->qij", 2.0 * wdet, eps, eps, optimize=True)
            K = (coef @ tt(T.reshape(nb, m * m))).reshape(-1, m, m)
            mu = coef
        self.B = tt(-np.einsum("q,qa,qj->aj", wdet, psi, div))
        self.M = tt(np.einsum("q,qa,qb->ab", wdet, psi, psi))
        self.Mmu = torch.einsum("cq,qab->cab", 1.0 / mu, tt(np.einsum("q,qa,qb->qab", wdet, psi, psi)))
        W = self.Mmu if c["schur"] == "P2" else self.M[None]
        self.G = c["gamma"] * (self.B.T @ torch.linalg.solve(W, self.B.expand(len(W), -1, -1)))
        self.K = K + self.G
        cells = _grid(n, dev)
        nn = [k * v + 1 for v in n]
        self.nn = nn
        stride = torch.tensor([1, nn[0], nn[0] * nn[1]][:d], device=dev)
        N = math.prod(nn)
        cn = ((k * cells[:, None, :] + torch.as_tensor(mi.copy(), device=dev)[None]) * stride).sum(-1)
        self.dofs = torch.cat([a * N + cn for a in range(d)], 1)
        self.freen = _free(n, k, dev)
        self.free = self.freen.repeat(d)
        self.nu = d * N
        if stars:
            self._stars(cells, stride, N, dev)

    def _scatter(self, v):
        return torch.zeros(self.nu, dtype=torch.float64, device=v.device).index_add_(0, self.dofs.reshape(-1), v.reshape(-1))

    def _mul(self, E, x):
        return self._scatter(torch.matmul(E, x[self.dofs][:, :, None])[..., 0])

    def apply(self, x):
        return self._mul(self.K, x * self.free) * self.free + x * ~self.free

    def al(self, x):
        return self._mul(self.G, x * self.free) * self.free

    def div(self, x):
        return ((x * self.free)[self.dofs] @ self.B.T).reshape(-1)

    def divt(self, p):
        return self._scatter(p.reshape(-1, self.npr) @ self.B) * self.free

    def _stars(self, cells, stride, N, dev):
        d, k, n = self.d, self.k, self.n
        w = 2 * k - 1
        off = _grid((w,) * d, dev)                                     # 0 .. 2k-2 per axis
        nv = [v + 1 for v in n]
        verts = _grid(nv, dev)
        node = k * verts[:, None, :] + off[None] - (k - 1)
        top = torch.tensor(self.nn, device=dev) - 1
        ok = ((node > 0) & (node < top)).all(-1)
        idx = (node.clamp(min=0).minimum(top) * stride).sum(-1)
        self.sdof = torch.cat([a * N + idx for a in range(d)], 1)
        self.sok = ok.repeat(1, d)
        S = torch.zeros(len(verts), d * w ** d, d * w ** d, dtype=torch.float64, device=dev)
        cstride = torch.tensor([1, n[0], n[0] * n[1]][:d], device=dev)
        nb = (k + 1) ** d
        for s in itertools.product(range(2), repeat=d):
            st = torch.tensor(s, device=dev)
            cell = verts - 1 + st
            vin = ((cell >= 0) & (cell < torch.tensor(n, device=dev))).all(-1).nonzero()[:, 0]
            loc = off - (k - 1) + k * (1 - st)                          # local node of each star offset
            lin = ((loc >= 0) & (loc <= k)).all(-1).nonzero()[:, 0]
            a = (loc[lin] * torch.tensor([1, k + 1, (k + 1) ** 2][:d], device=dev)).sum(-1)
            la = torch.cat([e * nb + a for e in range(d)])
            lo = torch.cat([e * w ** d + lin for e in range(d)])
            sub = self.K[(cell[vin] * cstride).sum(-1)][:, la][:, :, la]
            S[vin[:, None, None], lo[None, :, None], lo[None, None, :]] += sub
        both = self.sok[:, :, None] & self.sok[:, None, :]
        S = S * both + torch.diag_embed((~self.sok).double())
        self.sinv = torch.cat([torch.linalg.inv(part) for part in S.split(4096)])

    def star(self, r, sel=None):
        dof, ok, inv = (self.sdof, self.sok, self.sinv) if sel is None else (self.sdof[sel], self.sok[sel], self.sinv[sel])
        y = torch.matmul(inv, (r[dof] * ok)[:, :, None])[..., 0] * ok
        return torch.zeros_like(r).index_add_(0, dof.reshape(-1), y.reshape(-1))

    def interiors(self, r):
        """Local solves on the interiors of the next coarser level's cells."""
        v = 2 * _grid([m // 2 for m in self.n], r.device) + 1
        nv = [m + 1 for m in self.n]
        return self.star(r, (v * torch.tensor([1, nv[0], nv[0] * nv[1]][: self.d], device=r.device)).sum(-1))


def _p1(nc, k, dev):
    """Coarse order-k basis on nc cells at the nodes of 2 nc cells."""
    t = np.linspace(-1.0, 1.0, k + 1)
    P = np.zeros((2 * k * nc + 1, k * nc + 1))
    for f in range(2 * k * nc + 1):
        cell = min(f // (2 * k), nc - 1)
        x = 2.0 * (f - 2 * k * cell) / (2.0 * k) - 1.0
        for a in range(k + 1):
            P[f, k * cell + a] = np.prod([(x - t[b]) / (t[a] - t[b]) for b in range(k + 1) if b != a])
    return torch.as_tensor(P, device=dev)


class _Method:
    """The cycle and the solve on a hierarchy of _Ref levels."""

    def __init__(self, c, coef, mu, only_top=False):
        self.c = c
        sizes = _sizes(c)
        first = len(sizes) - 2 if only_top else 0
        self.lev = [None] * first + [_Ref(c, sizes[l], coef[l], mu[l] if mu else None,
                                          stars=l > 0 and not (only_top and l == first))
                                     for l in range(first, len(sizes))]
        if not only_top:
            f = self.lev[0].free.nonzero()[:, 0]
            eye = torch.zeros(self.lev[0].nu, device=f.device, dtype=torch.float64)
            cols = []
            for i in f.tolist():
                eye[i] = 1.0
                cols.append(self.lev[0].apply(eye)[f])
                eye[i] = 0.0
            self.cfree, self.chol = f, torch.linalg.cholesky(torch.stack(cols, 1))

    def _kron(self, l, x, transpose):
        hi, lo = self.lev[l], self.lev[l - 1]
        src = hi if transpose else lo
        x = (x * src.free).reshape([src.d] + list(reversed(src.nn)))
        for a in range(src.d):
            P = _p1(lo.n[a], lo.k, x.device)
            x = torch.movedim(torch.tensordot(x, P, dims=([x.dim() - 1 - a], [0 if transpose else 1])), -1, x.dim() - 1 - a)
        return x.reshape(-1) * (lo if transpose else hi).free

    def prolong(self, l, x):
        x = self._kron(l, x, False)
        return x if self.c.get("transfer") == "standard" else x - self.lev[l].interiors(self.lev[l].al(x))

    def restrict(self, l, r):
        if self.c.get("transfer") != "standard":
            r = r - self.lev[l].al(self.lev[l].interiors(r))
        return self._kron(l, r, True)

    def smooth(self, l, x, b):
        R = self.lev[l]
        if self.c.get("smoother") == "richardson":
            for _ in range(self.c["sweeps"]):
                x = x + 2.0 ** -R.d * R.star(b - R.apply(x))
            return x
        s = self.c["sweeps"]
        V, Z, H = [b - R.apply(x)], [], torch.zeros(s + 1, s, dtype=torch.float64, device=b.device)
        beta = V[0].norm()
        V[0] = V[0] / beta
        for j in range(s):
            Z.append(R.star(V[j]))
            w = R.apply(Z[j])
            Vm = torch.stack(V)
            h = Vm @ w
            w = w - h @ Vm
            H[: j + 1, j] = h
            H[j + 1, j] = w.norm()
            V.append(w / H[j + 1, j])
        e = torch.zeros(s + 1, 1, dtype=torch.float64, device=b.device)
        e[0] = beta
        y = torch.linalg.lstsq(H, e).solution[:, 0]
        return x + y @ torch.stack(Z)

    def cycle(self, b, l=None, x=None, f=None):
        l = len(self.lev) - 1 if l is None else l
        f = self.c.get("cycle") == "F" if f is None else f
        if l == 0:
            x = torch.zeros_like(b)
            x[self.cfree] = torch.cholesky_solve(b[self.cfree][:, None], self.chol)[:, 0]
            return x
        x = self.smooth(l, torch.zeros_like(b) if x is None else x, b)
        bc = self.restrict(l, b - self.lev[l].apply(x))
        e = self.cycle(bc, l - 1, None, f)
        if f and l > 1:
            e = self.cycle(bc, l - 1, e, False)
        return self.smooth(l, x + self.prolong(l, e), b)

    def solve(self, f):
        c, R = self.c, self.lev[-1]
        phi, wdet = (torch.as_tensor(v, dtype=torch.float64, device=f.device) for v in (R.phi, R.wdet))
        b1 = R._scatter(torch.einsum("q,cqa,qi->cai", wdet, f, phi).reshape(len(f), -1)) * R.free
        b = torch.cat([b1, torch.zeros(R.Mmu.shape[0] * R.npr, dtype=torch.float64, device=f.device)])
        inv = torch.linalg.inv(R.Mmu)
        S = inv + c["gamma"] * torch.linalg.inv(R.M) if c["schur"] == "P1" else (1.0 + c["gamma"]) * inv

        def prec(v):
            z1 = self.cycle(v[: R.nu])
            z2 = -torch.matmul(S, (v[R.nu:] - R.div(z1)).reshape(-1, R.npr, 1)).reshape(-1)
            x1 = z1 - self.cycle(R.divt(z2))
            z2[:: R.npr] -= z2[:: R.npr].mean()
            return torch.cat([x1, z2])

        beta, most = b.norm(), 290
        V, Z, H = [b / beta], [], np.zeros((most + 1, most))
        for k in range(most):
            Z.append(prec(V[k]))
            u, p = Z[k][: R.nu], Z[k][R.nu:]
            w = torch.cat([R.apply(u) + R.divt(p), R.div(u)])
            Vm = torch.stack(V)
            for _ in range(2):
                h = Vm @ w
                w = w - h @ Vm
                H[: k + 1, k] += h.cpu().numpy()
            H[k + 1, k] = float(w.norm())
            V.append(w / w.norm())
            e = np.zeros(k + 2)
            e[0] = float(beta)
            y, *_ = np.linalg.lstsq(H[: k + 2, : k + 1], e, rcond=None)
            if np.linalg.norm(e - H[: k + 2, : k + 1] @ y) <= 1e-13 * float(beta):
                break
        x = torch.as_tensor(y, device=f.device) @ torch.stack(Z)
        u, p = x[: R.nu], x[R.nu:].clone()
        p[:: R.npr] -= p[:: R.npr].mean()
        return u, p


def exact(case, seed):
    c = case
    if c["kind"] == "batch":
        out = []
        for i, s in enumerate(_batch_cases(c)):
            coef, _, _ = _problem(s, 1000 * seed + i)
            out.append(_Method(s, coef, None).cycle(_vector(_sizes(s)[-1], 2, 1000 * seed + i, torch.float32).double()))
        return out
    coef, mu, f = _problem(c, seed)
    if c["kind"] == "solve":
        u, p = _Method(c, coef, mu).solve(f)
        return {"u": u, "p": p}
    b = _vector(_sizes(c)[-1], c["order"], seed, _dtype(c)[0]).double()
    if c["kind"] == "cycle":
        return _Method(c, coef, mu).cycle(b)
    m, top = _Method(c, coef, mu, only_top=True), c["levels"] - 1
    xc = _vector(_sizes(c)[-2], c["order"], seed + 1, _dtype(c)[0]).double()
    return {"Ab": m.lev[top].apply(b), "Db": m.lev[top].star(b), "restricted": m.restrict(top, b),
            "prolonged": m.prolong(top, xc)}

"""Timed workloads: the calls a user of this package makes, over the sizes it is used at.

listed() names them; draw(rng) gives further ones of the same ranges.  A case is a dict
of plain values with a "kind":

  residual   Problem.residual: r = f - A x and ||r||^2 (every outer iteration's check)
  apply      Problem.apply: y = A x
  relax      Problem.relax: sweeps in place on A x = f (a smoother inside a user's own solver)
  cycle      Problem.precond: the hybrid cycle M (sweeps, then the trunk-basis correction)
             as the preconditioner of a user's own Krylov method
  solve      Problem.solve: FGMRES to a tolerance, or a few iterations of BiCGStab or
             FGMRES (a rounding difference of BiCGStab grows a hundredfold per iteration on
             these indefinite systems, so only its first iterations can be compared)
  many       solve_concurrent: problems of uneven size solved at once
  train      train.train_step: one Adam step of the DeepONet
  setup      Problem.don_load: trunk basis and coarse operator of a new problem

Mixed-precision (complex64) solves return complex128 storage; their results are handed
on as complex64, the precision they are computed in.
"""
import math

import numpy as np
import torch

import paper_2405_12380_gb300 as hm
from paper_2405_12380_gb300 import train as tr

LAYER = 8                     # absorbing-layer cells
STRENGTH = 0.5                # its strength


def listed():
    return [
        # the smallest call: the true residual of the 2D problem (64 x 64, k = 10)
        dict(name="residual-2d-64", kind="residual", dim=2, n=64, k0=10.0, dtype="c128", conj=False, field=False),
        # the residual on an odd grid (vertex-coarsened multigrid grids are odd), FP64, adjoint operator
        dict(name="residual-c128-129", kind="residual", dim=3, n=129, k0=32.0, dtype="c128", conj=True, field=False),
        # the complex64 operator on a grid larger than L2
        dict(name="apply-c64-256", kind="apply", dim=3, n=256, k0=32.0, dtype="c64", conj=False, field=False),
        # three complex64 red-black sweeps (one cycle's worth) on a grid larger than L2
        dict(name="relax-c64-256", kind="relax", dim=3, n=256, k0=32.0, dtype="c64", conj=False, field=False,
             relax="rbgs", sweeps=3, omega=1.0),
        # the adjoint workload's preconditioner: 96^3, a stored k^2 field, conjugate, FP64
        dict(name="cycle-field-96", kind="cycle", dim=3, n=96, k0=20.0, prec="fp64", conj=True, field=True,
             relax="rbgs", sweeps=3, omega=1.0, p=128, width=128, tau=1e-6),
        # the first BiCGStab iterations of the 64^3 FP64 workload (k = 16, p = 128)
        dict(name="bicgstab-fp64-64", kind="solve", dim=3, n=64, k0=16.0, prec="fp64", conj=False, field=False,
             method="bicgstab", relax="rbgs", sweeps=3, omega=1.0, p=128, width=128, tau=1e-6, tol=1e-14, maxit=4),
        # the first BiCGStab iterations of the 128^3 mixed-precision workload (k = 32, p = 256)
        dict(name="bicgstab-mixed-128", kind="solve", dim=3, n=128, k0=32.0, prec="mixed", conj=False, field=False,
             method="bicgstab", relax="rbgs", sweeps=3, omega=1.0, p=256, width=256, tau=1e-6, tol=1e-12, maxit=3),
        # the 2D workload solved to 1e-8: DeepONet-Jacobi (20 sweeps per correction) in
        # FGMRES(30), about a hundred steps of small launches
        dict(name="fgmres-2d-64", kind="solve", dim=2, n=64, k0=10.0, prec="fp64", conj=False, field=False,
             method="fgmres", relax="jacobi", sweeps=20, omega=0.6, p=32, width=64, tau=1e-6, tol=1e-8, maxit=2000),
        # eight problems of uneven size at once, mixed precision, six FGMRES(30) steps
        dict(name="many-mixed-8", kind="many", count=8, n_lo=48, n_hi=96, relax="rbgs", sweeps=3, omega=1.0, p=32,
             width=64, tau=1e-4, maxit=6),
        # one Adam step of the 64^3 DeepONet (batch 32, 16384 nodes per step), FP32
        dict(name="train-fp32-64", kind="train", dim=3, n=64, batch=32, nodes=16384, hidden=256, p=128, cores=False),
        # the same step with BF16 products on the tensor cores, a smaller grid and larger batch
        dict(name="train-bf16-40", kind="train", dim=3, n=40, batch=64, nodes=8192, hidden=256, p=128, cores=True),
        # trunk basis and coarse operator of a new 64^3 problem with its own k^2 field
        dict(name="setup-fp64-64", kind="setup", dim=3, n=64, k0=16.0, prec="fp64", field=True, p=128, width=128,
             tau=1e-3),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["residual", "apply", "relax", "relax", "cycle", "cycle", "solve", "solve", "many", "train",
                       "train", "setup"])
    if kind in ("residual", "apply", "relax"):
        dim = rng.choice([2, 3, 3])
        n = _log_int(rng, 33, 1024) if dim == 2 else _log_int(rng, 17, 256)
        c = dict(kind=kind, dim=dim, n=n, k0=round(rng.uniform(8, 32), 2), dtype=rng.choice(["c64", "c128"]),
                 conj=rng.random() < 0.3, field=rng.random() < 0.25)
        if kind == "relax":
            relax = rng.choice(["jacobi", "rbgs", "rbgs", "sor", "ssor"])
            c.update(relax=relax, sweeps=rng.randint(1, 4), omega=0.6 if relax == "jacobi" else 1.2)
        return c
    if kind in ("cycle", "solve"):
        dim = rng.choice([2, 3, 3])
        n = _log_int(rng, 33, 256) if dim == 2 else _log_int(rng, 33, 128)
        p = rng.choice([32, 64, 128])
        relax = rng.choice(["jacobi", "rbgs", "rbgs"])
        c = dict(kind=kind, dim=dim, n=n, k0=round(rng.uniform(8, 32), 2), prec=rng.choice(["fp64", "mixed"]),
                 conj=rng.random() < 0.3, field=rng.random() < 0.3, relax=relax, sweeps=rng.randint(1, 4),
                 omega=0.6, p=p, width=p, tau=rng.choice([1e-4, 1e-6]))
        if kind == "solve":
            if c["prec"] == "fp64" and rng.random() < 0.6:
                c.update(method="bicgstab", tol=1e-14, maxit=rng.randint(1, 3))
            else:
                c.update(method="fgmres", tol=1e-14, maxit=rng.randint(3, 8 if c["prec"] == "mixed" else 20))
        return c
    if kind == "many":
        lo = rng.randint(33, 64)
        return dict(kind="many", count=rng.randint(3, 10), n_lo=lo, n_hi=rng.randint(lo + 8, 100), relax="rbgs",
                    sweeps=rng.randint(1, 3), omega=1.0, p=32, width=64, tau=1e-4, maxit=rng.randint(3, 8))
    if kind == "train":
        dim = rng.choice([2, 3])
        n = _log_int(rng, 32, 300) if dim == 2 else _log_int(rng, 16, 64)
        return dict(kind="train", dim=dim, n=n, batch=rng.randint(8, 96), nodes=min(_log_int(rng, 512, 16384), n ** dim),
                    hidden=rng.choice([100, 128, 256]), p=rng.choice([32, 64, 100, 128]), cores=rng.random() < 0.4)
    return dict(kind="setup", dim=3, n=_log_int(rng, 21, 72), k0=round(rng.uniform(8, 24), 2),
                prec=rng.choice(["fp64", "mixed"]), field=True, p=rng.choice([32, 64, 128]),
                width=rng.choice([64, 128]), tau=1e-3)


# ------------------------------------------------------------------------- inputs
_DEV = "cuda"


def _gen(seed, salt=0):
    return torch.Generator(device=_DEV).manual_seed(int(seed) * 1000 + salt)


def _cnormal(N, g, dtype=torch.complex128):
    return torch.randn(N, generator=g, device=_DEV, dtype=torch.complex128).to(dtype)


def _axes(dim, n):
    i = torch.arange(n, device=_DEV)
    if dim == 2:
        return i[None, :], i[:, None]
    return i[None, None, :], i[None, :, None], i[:, None, None]


def _mask(dim, n, sphere=False):
    """1 on the outer ring and on a centred scatterer (a cube of a quarter of the domain's
    side, or a sphere), as uint8 of N entries."""
    ax = _axes(dim, n)
    m = torch.zeros((n,) * dim, dtype=torch.bool, device=_DEV)
    w = max(2, n // 4)
    lo = (n - w) // 2
    box = torch.ones_like(m)
    r2 = torch.zeros((n,) * dim, device=_DEV, dtype=torch.float64)
    for a in ax:
        m |= (a == 0) | (a == n - 1)
        box &= (a >= lo) & (a < lo + w)
        r2 = r2 + ((a.double() / (n - 1)) - 0.5) ** 2
    m |= (r2 <= 0.12 ** 2) if sphere else box
    return m.reshape(-1).to(torch.uint8)


def _field(dim, n, k0, g):
    """k^2 of an adjoint iteration: the absorbing layer times a smooth random perturbation (5%)."""
    h = 1.0 / (n - 1)
    scale = torch.ones((n,) * dim, device=_DEV, dtype=torch.float64)
    eta = torch.zeros((n,) * dim, device=_DEV, dtype=torch.float64)
    for a in _axes(dim, n):
        eta = torch.maximum(eta, (LAYER - torch.minimum(a, n - 1 - a)).clamp(min=0) / LAYER)
    for _ in range(8):
        c = 0.2 + 0.6 * torch.rand(dim, generator=g, device=_DEV, dtype=torch.float64)
        r2 = sum((a * h - c[q]) ** 2 for q, a in enumerate(_axes(dim, n)))
        amp = 0.1 * torch.rand(1, generator=g, device=_DEV, dtype=torch.float64) - 0.05
        scale = scale + amp * torch.exp(-r2 / (2 * 0.08 ** 2))
    base = k0 * k0 * scale
    return torch.complex(base, base * (STRENGTH * eta * eta)).reshape(-1)


def _source(dim, n, mask, g, sigma=0.05):
    """A complex Gaussian source at a random point off the scatterer, zero on Dirichlet nodes."""
    h = 1.0 / (n - 1)
    lo = LAYER * h + sigma
    c = lo + (1 - 2 * lo) * torch.rand(dim, generator=g, device=_DEV, dtype=torch.float64)
    c[0] = torch.where(c[0] > 0.5, c[0].clamp(min=min(0.75, 1 - lo)), c[0].clamp(max=max(0.25, lo)))
    r2 = sum((a * h - c[q]) ** 2 for q, a in enumerate(_axes(dim, n)))
    ph = 2 * math.pi * torch.rand(1, generator=g, device=_DEV, dtype=torch.float64)
    s = (torch.exp(-r2 / (2 * sigma * sigma)) * torch.exp(1j * ph)).reshape(-1)
    return torch.where(mask == 1, torch.zeros_like(s), s)


def _trunk(dim, width, p, seed):
    """Glorot-normal trunk [dim, width, width, p], zero biases."""
    rng = np.random.default_rng(seed)
    ws = [dim, width, width, p]
    return [(rng.standard_normal((b, a)) * math.sqrt(2.0 / (a + b)), np.zeros(b)) for a, b in zip(ws[:-1], ws[1:])]


def _problem(c, seed):
    dim, n = c["dim"], c["n"]
    mask = _mask(dim, n)
    k2 = _field(dim, n, c["k0"], _gen(seed, 1)) if c.get("field") else None
    prec = c.get("prec") or ("mixed" if c["dtype"] == "c64" else "fp64")
    return hm.Problem(dim, n, c["k0"], mask, layer_cells=LAYER, layer_strength=STRENGTH, k2=k2, precision=prec), mask


def _sizes(c):
    """The uneven grid sizes and wavenumbers of a "many" case."""
    rng = np.random.default_rng(c["count"] * 1000 + c["n_lo"])
    out = []
    for _ in range(c["count"]):
        n = int(rng.integers(c["n_lo"], c["n_hi"] + 1))
        out.append((n, float(rng.uniform(8.0, min(32.0, 0.2 * math.pi * (n - 1))))))
    return out


def _net(c, seed):
    """DeepONet in mid-training: Glorot weights and Adam moments of gradients seen before."""
    g = _gen(seed, 2)
    N = c["n"] ** c["dim"]

    def layers(ws):
        out = []
        for a, b in zip(ws[:-1], ws[1:]):
            l = tr.Layer(torch.randn(b, a, generator=g, device=_DEV) * math.sqrt(2.0 / (a + b)),
                         0.01 * torch.randn(b, generator=g, device=_DEV))
            for m, v, like in (("mW", "vW", l.W), ("mb", "vb", l.b)):
                setattr(l, m, 1e-4 * torch.randn(like.shape, generator=g, device=_DEV))
                setattr(l, v, 1e-7 + 1e-6 * torch.rand(like.shape, generator=g, device=_DEV))
            out.append(l)
        return out

    net = tr.DeepONet(layers([2 * N, c["hidden"], c["hidden"], 2 * c["p"]]),
                      layers([c["dim"], c["hidden"], c["hidden"], c["p"]]), step=100)
    X = torch.randn(c["batch"], 2 * N, generator=g, device=_DEV)
    Y = torch.randn(c["batch"], 2 * c["nodes"], generator=g, device=_DEV)
    Xc = torch.rand(c["nodes"], c["dim"], generator=g, device=_DEV)
    return net, X, Xc, Y


def prepare(case, seed):
    c, kind = case, case["kind"]
    if kind == "train":
        net, X, Xc, Y = _net(c, seed)
        return dict(kind=kind, net=net, X=X, Xc=Xc, Y=Y, cores=c["cores"])
    if kind == "many":
        Ps, fs = [], []
        for q, (n, k0) in enumerate(_sizes(c)):
            mask = _mask(3, n, sphere=q % 2 == 1)
            P = hm.Problem(3, n, k0, mask, layer_cells=LAYER, layer_strength=STRENGTH, precision="mixed")
            P.don_load(_trunk(3, c["width"], c["p"], q), c["p"], tau=c["tau"])
            Ps.append(P)
            fs.append(_source(3, n, mask, _gen(seed, 10 + q), 0.04))
        o = hm.opts("fgmres", c["relax"], c["sweeps"], omega=c["omega"], tol=1e-14, restart=30, maxit=c["maxit"])
        return dict(kind=kind, P=Ps, f=fs, o=o)
    P, mask = _problem(c, seed)
    N, g = P.N, _gen(seed, 3)
    if kind == "setup":
        return dict(kind=kind, P=P, layers=_trunk(3, c["width"], c["p"], 0), p=c["p"], tau=c["tau"])
    if kind in ("residual", "apply", "relax"):
        dt = torch.complex64 if c["dtype"] == "c64" else torch.complex128
        x = _cnormal(N, g, dt)
        f = (c["n"] - 1) ** 2 * _cnormal(N, g, dt)          # the scale of A x
        f = torch.where(mask == 1, x, f)
        return dict(kind=kind, P=P, x=x, f=f, conj=c["conj"], relax=c.get("relax"), sweeps=c.get("sweeps"),
                    omega=c.get("omega"))
    P.don_load(_trunk(c["dim"], c["width"], c["p"], 0), c["p"], tau=c["tau"])
    o = hm.opts(c.get("method", "bicgstab"), c["relax"], c["sweeps"], omega=c["omega"], tol=c.get("tol", 1e-8),
                restart=30, maxit=c.get("maxit", 1), conj=c["conj"])
    if kind == "cycle":
        r = _cnormal(N, g)
        return dict(kind=kind, P=P, r=torch.where(mask == 1, torch.zeros_like(r), r), o=o, mixed=c["prec"] == "mixed")
    return dict(kind=kind, P=P, f=_source(c["dim"], c["n"], mask, g), o=o, mixed=c["prec"] == "mixed")


def run(state):
    s, kind = state, state["kind"]
    if kind == "residual":
        return s["P"].residual(s["f"], s["x"], conj=s["conj"])
    if kind == "apply":
        return s["P"].apply(s["x"], conj=s["conj"])
    if kind == "relax":
        return s["P"].relax(s["relax"], s["f"], s["x"], sweeps=s["sweeps"], omega=s["omega"], conj=s["conj"])
    if kind == "cycle":
        z = s["P"].precond(s["r"], s["o"])
        return z.to(torch.complex64) if s["mixed"] else z
    if kind == "solve":
        x = s["P"].solve(s["f"], None, s["o"])[0]
        return x.to(torch.complex64) if s["mixed"] else x
    if kind == "many":
        return [x.to(torch.complex64) for x in hm.solve_concurrent(s["P"], s["f"], None, s["o"])[0]]
    if kind == "setup":
        s["P"].don_load(s["layers"], s["p"], tau=s["tau"])
        return s["P"].basis(), s["P"].coarse_inverse()
    tr.set_tensor_cores(s["cores"])
    loss = tr.train_step(s["net"], s["X"], s["Xc"], s["Y"], lr=1e-4)
    tr.set_tensor_cores(False)
    net = s["net"]
    return dict(loss=loss, **{part: [(l.W, l.b, l.gW, l.gb) for l in getattr(net, part)] for part in ("branch", "trunk")})


# --------------------------------------------------------------------- algorithmic work
def _kept(dim, p, tau):
    """About how many trunk columns the selection keeps (seeded trunks, width >= 64)."""
    d = -math.log10(tau)
    return int(min(p, 2 * d ** 1.8 if dim == 3 else d ** 1.6))


def _cycle_work(N, dim, k, prec, sweeps):
    """One hybrid cycle: r in, z out, two table bytes a node, the basis once."""
    cb, qb = (8, 2) if prec == "mixed" else (16, 8)
    return N * (2 * cb + 2 + qb * k), N * (sweeps * (4 * dim + 12) + 4 * dim + 8 + 6 * k)


def work(case):
    c, kind = case, case["kind"]
    if kind == "many":
        b = f = 0.0
        for n, _ in _sizes(c):
            cb, cf = _cycle_work(n ** 3, 3, _kept(3, c["p"], c["tau"]), "mixed", c["sweeps"])
            it = c["maxit"]
            # per step the cycle, the operator and the orthogonalisation against j FP64 vectors
            b += it * (cb + n ** 3 * 16) + n ** 3 * 16 * it * (it + 1)
            f += it * (cf + n ** 3 * 30) + n ** 3 * 16 * it * (it + 1)
        return dict(bytes=b, flops=f)
    N = c["n"] ** c["dim"]
    if kind == "train":
        B, P, H, p = c["batch"], c["nodes"], c["hidden"], c["p"]
        wb = 2 * N * H + H * H + H * 2 * p
        wt = c["dim"] * H + H * H + H * p
        # weights read forward and backward, gradients out, Adam's p, m, v in and out
        return dict(bytes=4.0 * ((wb + wt) * 8 + B * (2 * N + 2 * P) + P * c["dim"]),
                    flops=2.0 * B * (2 * (2 * N * H) + 3 * (H * H + H * 2 * p)) + 2.0 * P * (3 * wt) + 2.0 * 6 * B * P * p)
    if kind == "setup":
        k, w, p = _kept(3, c["p"], c["tau"]), c["width"], c["p"]
        return dict(bytes=8.0 * N * k * 2, flops=N * (2.0 * (3 * w + w * w + w * p) + 1.0 * p * p + 2.0 * k * k + 4.0 * k * k))
    cb = 8 if c.get("dtype") == "c64" else 16
    if kind in ("residual", "apply", "relax"):
        extra = cb if c["field"] else 0
        vecs = {"residual": 3, "apply": 2, "relax": 3}[kind]
        return dict(bytes=N * (vecs * cb + 2.0 + extra), flops=N * (4.0 * c["dim"] + 10) * (c.get("sweeps") or 1))
    k = _kept(c["dim"], c["p"], c["tau"])
    b, f = _cycle_work(N, c["dim"], k, c["prec"], c["sweeps"])
    if kind == "cycle":
        return dict(bytes=float(b), flops=float(f))
    vb = 8 if c["prec"] == "mixed" else 16
    if c["method"] == "bicgstab":
        it = c["maxit"]
        # two cycles, two operators and the vector updates (x, r, p, v, s, t) an iteration
        return dict(bytes=float(it * (2 * b + N * vb * 14)), flops=float(it * (2 * f + N * (2 * (4 * c["dim"] + 10) + 60))))
    it = c["maxit"] if c["tol"] < 1e-12 else 100
    m = min(it, 30)
    return dict(bytes=float(it * (b + N * 16 * 2) + it * N * 16 * (m + 1)),
                flops=float(it * (f + N * (4 * c["dim"] + 10)) + it * N * 8 * (m + 1)))


# ------------------------------------------------------------------ plain 64-bit results
class _Op:
    """The operator, sweeps, trunk basis and cycle in plain FP64 torch."""

    def __init__(self, dim, n, k0, mask, k2=None, conj=False):
        self.dim, self.n, self.h2 = dim, n, float((n - 1) ** 2)
        self.shape = (n,) * dim
        self.fluid = (mask == 0).reshape(self.shape)
        if k2 is None:
            eta = torch.zeros(self.shape, device=_DEV, dtype=torch.float64)
            for a in _axes(dim, n):
                eta = torch.maximum(eta, (LAYER - torch.minimum(a, n - 1 - a)).clamp(min=0) / LAYER)
            k2 = torch.complex(torch.full_like(eta, k0 * k0), k0 * k0 * STRENGTH * eta * eta)
        k2 = k2.reshape(self.shape)
        self.diag = (k2.conj() if conj else k2) - 2.0 * dim * self.h2
        self.red = (sum(_axes(dim, n)) % 2) == 0

    def nbrs(self, x):
        u = torch.where(self.fluid, x, torch.zeros_like(x))
        s = torch.zeros_like(u)
        for ax in range(self.dim):
            s.narrow(ax, 1, self.n - 1).add_(u.narrow(ax, 0, self.n - 1))
            s.narrow(ax, 0, self.n - 1).add_(u.narrow(ax, 1, self.n - 1))
        return s

    def apply(self, x):
        x = x.reshape(self.shape)
        return torch.where(self.fluid, self.h2 * self.nbrs(x) + self.diag * x, x).reshape(-1)

    def sweeps(self, kind, omega, count, f, x):
        f, x = f.reshape(self.shape), x.reshape(self.shape)
        if kind == "rbgs":
            omega = 1.0
        for _ in range(count):
            for colour in {"jacobi": (None,), "ssor": (0, 1, 1, 0)}.get(kind, (0, 1)):
                new = torch.where(self.fluid, (f - self.h2 * self.nbrs(x)) / self.diag, f)
                step = x + omega * (new - x)
                x = step if colour is None else torch.where(self.red == (colour == 0), step, x)
        return x.reshape(-1)

    def basis(self, layers, p, tau, bf16=False):
        """Columns kept in natural order (classical Gram-Schmidt twice), Q and (Q^T A Q)^-1."""
        h = 1.0 / (self.n - 1)
        z = torch.stack([(a * h).expand(self.shape).reshape(-1) for a in _axes(self.dim, self.n)], 1).double()
        for q, (W, b) in enumerate(layers):
            z = z @ torch.from_numpy(W).to(_DEV).T + torch.from_numpy(b).to(_DEV)
            z = torch.tanh(z) if q < len(layers) - 1 else z
        T = torch.where(self.fluid.reshape(-1, 1), z[:, :p], torch.zeros(1, device=_DEV, dtype=torch.float64)).T.contiguous()
        Q = torch.empty_like(T)
        k = 0
        for j in range(p):
            v = T[j].clone()
            for _ in range(2):
                v -= Q[:k].T @ (Q[:k] @ v)
            if float(v.norm()) > tau * float(T[j].norm()):
                Q[k] = v / v.norm()
                k += 1
        Q = Q[:k].clone()
        if bf16:
            Q = Q.float().bfloat16().double()
        self.Q = Q
        AQ = torch.stack([self.apply(q.to(torch.complex128)) for q in Q])
        self.Ac = torch.complex(Q @ AQ.real.T, Q @ AQ.imag.T)
        return self

    def cycle(self, kind, omega, count, r):
        z = self.sweeps(kind, omega, count, r, torch.zeros_like(r))
        v = r - self.apply(z)
        c = torch.complex(self.Q @ v.real, self.Q @ v.imag)
        y = torch.linalg.solve(self.Ac, c)
        return z + torch.complex(self.Q.T @ y.real, self.Q.T @ y.imag)

    def bicgstab(self, M, f, its):
        x = torch.zeros_like(f)
        r = f - self.apply(x)
        rh, p, v = r.clone(), torch.zeros_like(r), torch.zeros_like(r)
        rho = al = om = torch.ones((), device=_DEV, dtype=torch.complex128)
        for _ in range(its):
            rn = torch.vdot(rh, r)
            p = r + (rn / rho) * (al / om) * (p - om * v)
            rho, ph = rn, M(p)
            v = self.apply(ph)
            al = rho / torch.vdot(rh, v)
            s = r - al * v
            sh = M(s)
            t = self.apply(sh)
            om = torch.vdot(t, s) / torch.vdot(t, t)
            x, r = x + al * ph + om * sh, s - om * t
        return x

    def fgmres(self, M, f, its):
        """`its` <= 30 steps from zero (one cycle)."""
        beta = f.norm()
        V, Z, H = [f / beta], [], torch.zeros(its + 1, its, dtype=torch.complex128, device=_DEV)
        for j in range(its):
            Z.append(M(V[j]))
            w = self.apply(Z[j])
            for _ in range(2):
                for i in range(j + 1):
                    hij = torch.vdot(V[i], w)
                    w = w - hij * V[i]
                    H[i, j] += hij
            H[j + 1, j] = w.norm()
            V.append(w / w.norm())
        e = torch.zeros(its + 1, 1, dtype=torch.complex128, device=_DEV)
        e[0] = beta
        y = torch.linalg.lstsq(H.cpu(), e.cpu()).solution.to(_DEV)
        return sum(y[j] * Z[j] for j in range(its))

    def dense_solve(self, f):
        N = self.n ** self.dim
        A = torch.stack([self.apply(col) for col in torch.eye(N, dtype=torch.complex128, device=_DEV)], 1)
        return torch.linalg.solve(A, f)


def _exact_train(c, seed):
    net, X, Xc, Y = _net(c, seed)
    d = torch.float64
    X, Xc, Y = X.to(d), Xc.to(d), Y.to(d)
    br = [(l.W.to(d).requires_grad_(), l.b.to(d).requires_grad_()) for l in net.branch]
    tk = [(l.W.to(d).requires_grad_(), l.b.to(d).requires_grad_()) for l in net.trunk]

    def mlp(x, layers, act):
        for q, (W, b) in enumerate(layers):
            x = x @ W.T + b
            x = act(x) if q < len(layers) - 1 else x
        return x

    p = c["p"]
    B, T = mlp(X, br, torch.relu), mlp(Xc, tk, torch.tanh)
    pred = torch.cat([B[:, :p] @ T.T, B[:, p:] @ T.T], 1)
    loss = ((pred - Y) ** 2).sum(1) / (Y ** 2).sum(1)
    loss.mean().backward()
    t = net.step + 1

    def adam(w, m, v):
        g = w.grad
        m, v = 0.9 * m.to(d) + 0.1 * g, 0.999 * v.to(d) + 0.001 * g * g
        return (w - 1e-4 * (m / (1 - 0.9 ** t)) / ((v / (1 - 0.999 ** t)).sqrt() + 1e-8)).detach()

    out = {}
    for part, ws in (("branch", br), ("trunk", tk)):
        out[part] = [(adam(W, l.mW, l.vW), adam(b, l.mb, l.vb), W.grad, b.grad)
                     for l, (W, b) in zip(getattr(net, part), ws)]
    return dict(loss=loss.detach(), **out)


def exact(case, seed):
    c, kind = case, case["kind"]
    if kind == "train":
        return _exact_train(c, seed)
    if kind == "many":
        out = []
        for q, (n, k0) in enumerate(_sizes(c)):
            mask = _mask(3, n, sphere=q % 2 == 1)
            op = _Op(3, n, k0, mask).basis(_trunk(3, c["width"], c["p"], q), c["p"], c["tau"], bf16=True)
            out.append(op.fgmres(lambda r: op.cycle(c["relax"], c["omega"], c["sweeps"], r),
                                 _source(3, n, mask, _gen(seed, 10 + q), 0.04), c["maxit"]))
        return out
    dim, n = c["dim"], c["n"]
    mask = _mask(dim, n)
    k2 = _field(dim, n, c["k0"], _gen(seed, 1)) if c.get("field") else None
    op, g, N = _Op(dim, n, c["k0"], mask, k2, c.get("conj", False)), _gen(seed, 3), n ** dim
    if kind == "setup":
        op.basis(_trunk(3, c["width"], c["p"], 0), c["p"], c["tau"], bf16=c["prec"] == "mixed")
        return op.Q.T.contiguous(), torch.linalg.inv(op.Ac)
    if kind in ("residual", "apply", "relax"):
        dt = torch.complex64 if c["dtype"] == "c64" else torch.complex128
        x = _cnormal(N, g, dt)
        f = (n - 1) ** 2 * _cnormal(N, g, dt)
        f = torch.where(mask == 1, x, f).to(torch.complex128)
        x = x.to(torch.complex128)
        if kind == "apply":
            return op.apply(x)
        if kind == "relax":
            return op.sweeps(c["relax"], c["omega"], c["sweeps"], f, x)
        r = f - op.apply(x)
        return r, (r.abs() ** 2).sum().reshape(1)
    # at tau = 1e-6 the columns kept on a large grid hang on rounding (the Gram matrix's
    # error over tau^2), so a plain result in another basis says nothing there
    if c["tau"] < 1e-5 and n > (64 if dim == 3 else 100):
        return None
    if kind == "solve" and c["method"] == "fgmres" and c["tol"] > 1e-12:
        return op.dense_solve(_source(dim, n, mask, g)) if N <= 5000 else None
    op.basis(_trunk(dim, c["width"], c["p"], 0), c["p"], c["tau"], bf16=c["prec"] == "mixed")
    M = lambda r: op.cycle(c["relax"], c["omega"], c["sweeps"], r)  # noqa: E731
    if kind == "cycle":
        r = _cnormal(N, g)
        return M(torch.where(mask == 1, torch.zeros_like(r), r))
    f = _source(dim, n, mask, g)
    return (op.bicgstab if c["method"] == "bicgstab" else op.fgmres)(M, f, c["maxit"])

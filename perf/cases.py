"""Performance cases: what users of the library have it do, at the sizes they do it.

Every case goes through the public Python entry points (Solver, VCycleFn,
learn.Problem, the mlp_* calls) on inputs that problems.py generates.  Eight
kinds of work, each a `what` of a case:

  smooth    one smoother application on the finest level
  vcycle    one V-cycle z = B r (the preconditioner of a caller's own solver)
  pcg       a whole preconditioned CG solve
  grad      V-cycle forward and backward through torch.autograd
  train     loss and weight gradient of one training problem
  mlp       forward, backward and Adam step of the weight-predicting network
  sa_pcg    a solve on a smoothed-aggregation hierarchy (30 coarse sweeps,
            one-reduction flexible CG)
  sa_setup  a smoothed-aggregation hierarchy built on the device (host CSR in,
            host CSR out)

exact() restates the method on 7-point stencils (and, for smoothed
aggregation, on torch sparse matrices) in 64-bit torch.
"""
import functools
import math

import numpy as np
import torch

from paper_2407_09848_gb300 import amgps, learn
from paper_2407_09848_gb300 import problems as pr
from paper_2407_09848_gb300.amgps import Solver
from paper_2407_09848_gb300.autograd import VCycleFn

COARSE_MAX = 512
# published optimal 4th-kind weights and 1st-kind interval ends by degree
BETA = {2: (1.0238728757031317, 1.2640890537108553),
        3: (1.008425447820283, 1.0886783920873089, 1.3375312590961856),
        4: (1.0039131042728535, 1.0403581118859304, 1.1486349854625488, 1.382688692410006),
        6: (1.0012851725594023, 1.0130429303523336, 1.0467821512411335, 1.1161648941967548,
            1.2382902021844457, 1.4352429710674486)}
ASTAR = {2: 0.18053599274030066, 3: 0.11592784648622129, 4: 0.08207806595903835,
         6: 0.048660582342606194}


def listed():
    return [
        # one application of the default smoother on the smallest configured
        # grid: what a caller's own multigrid pays per call
        dict(name="smooth_32", what="smooth", nx=32, ny=32, nz=32, problem="poisson", prec="f64",
             kind="cheb4_opt", degree=4, zero=True),
        # the 1st-kind polynomial at a higher degree on a ragged anisotropic
        # grid, from a given start: a stand-alone smoother sweep
        dict(name="smooth_ragged", what="smooth", nx=173, ny=151, nz=129, problem="aniso",
             prec="f64", kind="cheb1_opt", degree=6, zero=False),
        # one V-cycle on a small odd variable-coefficient grid: the library as
        # a preconditioner inside a caller's Krylov method
        dict(name="vcycle_odd", what="vcycle", nx=61, ny=53, nz=47, problem="varcoef",
             prec="f64", kind="cheb4_opt", degree=4),
        # the smallest configured solve (32^3 Poisson to 1e-8)
        dict(name="pcg_32", what="pcg", nx=32, ny=32, nz=32, problem="poisson", prec="f64",
             kind="cheb4_opt", degree=4, outer="cg"),
        # an ordinary variable-coefficient solve with FP32 matrix values
        dict(name="pcg_f32_128", what="pcg", nx=128, ny=128, nz=128, problem="varcoef",
             prec="f32", kind="cheb4_opt", degree=4, outer="flexible"),
        # inference at scale: BF16 matrix values, per-level weights, anisotropic
        dict(name="pcg_bf16_192", what="pcg", nx=192, ny=192, nz=192, problem="aniso",
             prec="bf16", kind="weights", degree=4, outer="cg"),
        # the headline: 256^3 Poisson, FP64, optimal 4th kind of degree 4
        dict(name="pcg_256", what="pcg", nx=256, ny=256, nz=256, problem="poisson", prec="f64",
             kind="cheb4_opt", degree=4, outer="cg"),
        # differentiating through the V-cycle (learned weights per level)
        dict(name="grad_odd", what="grad", nx=97, ny=81, nz=72, problem="varcoef", degree=4),
        # one training problem's loss and gradient: 64^3, 32 error vectors
        dict(name="train_64", what="train", nx=64, ny=64, nz=64, problem="varcoef", m=32),
        # the network's step on the levels of a minibatch of 16 such problems
        dict(name="mlp_48", what="mlp", batch=48),
        # the paper's solver setting on smoothed aggregation
        dict(name="sa_pcg_96", what="sa_pcg", nx=96, ny=96, nz=96, kind="cheb4_opt", degree=4),
        # setting such a hierarchy up from the fine matrix
        dict(name="sa_setup_64", what="sa_setup", nx=64, ny=64, nz=64),
    ]


def _grid(rng, lo, hi):
    """Three edge lengths (odd ones among them) around one log-uniform size."""
    base = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    return dict(zip(("nx", "ny", "nz"),
                    (max(lo, min(hi, round(base * rng.uniform(0.8, 1.2)))) for _ in range(3))))


def draw(rng):
    what = rng.choice(["smooth", "vcycle", "pcg", "pcg", "grad", "train", "mlp", "sa_pcg",
                       "sa_setup"])
    if what == "mlp":
        return dict(what=what, batch=round(math.exp(rng.uniform(math.log(3), math.log(2048)))))
    if what == "train":
        return dict(what=what, problem="varcoef", m=rng.randint(3, 32), **_grid(rng, 20, 64))
    if what == "sa_setup":
        return dict(what=what, **_grid(rng, 20, 72))
    degree = rng.choice([2, 3, 4, 6])
    if what == "sa_pcg":
        return dict(what=what, kind=rng.choice(["cheb4_opt", "cheb1_opt", "l1jacobi"]),
                    degree=degree, **_grid(rng, 24, 96))
    problem = rng.choice(["poisson", "varcoef", "aniso"])
    if what == "grad":
        return dict(what=what, problem=problem, degree=degree, **_grid(rng, 24, 112))
    c = dict(what=what, problem=problem, prec=rng.choice(["f64", "f64", "f32", "bf16"]),
             kind=rng.choice(["cheb4_opt", "cheb4", "cheb1_opt", "weights", "l1jacobi"]),
             degree=degree)
    if what == "smooth":
        c.update(zero=rng.random() < 0.5)
    if what == "pcg":
        c.update(outer=rng.choice(["cg", "cg", "flexible", "fcg1"]))
    c.update(_grid(rng, 24, 176 if what == "smooth" else 128))
    return c


# ---- inputs -----------------------------------------------------------------

def _stencil(case, seed):
    n = dict(nx=case["nx"], ny=case["ny"], nz=case["nz"])
    if case.get("problem", "poisson") == "poisson":
        return pr.poisson(**n)
    if case["problem"] == "aniso":
        return pr.aniso(eps=1e-3, **n)
    return pr.varcoef(sigma=1.0, ell=8.0, seed=seed, **n)


@functools.lru_cache(maxsize=6)
def _constant_hierarchy(problem, nx, ny, nz):
    # a constant-coefficient matrix is the same for every right-hand side
    return pr.build_hierarchy(_stencil(dict(problem=problem, nx=nx, ny=ny, nz=nz), 0), COARSE_MAX)


def _hierarchy(case, seed):
    if case["problem"] == "varcoef":
        return pr.build_hierarchy(_stencil(case, seed), COARSE_MAX)
    return _constant_hierarchy(case["problem"], case["nx"], case["ny"], case["nz"])


@functools.lru_cache(maxsize=4)
def _constant_sa(nx, ny, nz):
    st = pr.poisson(nx, ny, nz)
    builder = Solver()
    As, Ps, _ = builder.sa_hierarchy(pr.to_csr(st), pr.geometric_aggregates(st.shape, COARSE_MAX))
    builder.close()
    return As, Ps


def _levels(case):
    """Grid shapes (nz, ny, nx) of the hierarchy, the coarsest last."""
    out = [(case["nz"], case["ny"], case["nx"])]
    while math.prod(out[-1]) > COARSE_MAX and min(out[-1]) >= 2:
        out.append(tuple((s + 1) // 2 for s in out[-1]))
    return out


def _n(case):
    return case["nx"] * case["ny"] * case["nz"]


def _weights(case, seed):
    """Per-level weights near the optimal ones, as a trained network gives."""
    g = np.random.default_rng(seed + 1)
    k = case["degree"]
    nl = len(_levels(case)) - 1
    return np.asarray(BETA[k]) * (1.0 + 0.02 * g.uniform(-1.0, 1.0, (nl, k)))


def _vec(seed, *shape, normal=False):
    g = torch.Generator(device="cuda").manual_seed(seed)
    if normal:
        return torch.randn(shape, generator=g, dtype=torch.float64, device="cuda")
    return torch.rand(shape, generator=g, dtype=torch.float64, device="cuda") * 2.0 - 1.0


def _mlp_inputs(case, seed):
    g = np.random.default_rng(seed)
    B = case["batch"]
    net = learn.WeightMLP(seed=seed)
    th = net.params.cpu().numpy()
    th[4736:4992] = 0.1 * g.standard_normal(256)  # W3: a network in training
    net.params = torch.from_numpy(th).cuda()
    feats = g.uniform(0.0, 1.0, (B, 8)).astype(np.float32)
    gbeta = (g.standard_normal((B, 4)) / B).astype(np.float32)
    return net, feats, gbeta


def _set(S, case, seed):
    if case["kind"] == "weights":
        for l, w in enumerate(_weights(case, seed)):
            S.set_smoother(l, "weights", case["degree"], weights=w)
    else:
        S.set_smoother(-1, case["kind"], case["degree"])


def prepare(case, seed):
    what = case["what"]
    s = dict(case=case)
    if what == "mlp":
        net, feats, gbeta = _mlp_inputs(case, seed)
        s.update(net=net, feats=feats, gbeta=gbeta)
    elif what == "sa_setup":
        # the fine matrix scaled by a seeded constant
        st = pr.poisson(case["nx"], case["ny"], case["nz"])
        A = pr.to_csr(st) * (1.0 + np.random.default_rng(seed).random())
        s.update(S=Solver(), A=A, levels=pr.geometric_aggregates(st.shape, COARSE_MAX))
    elif what == "sa_pcg":
        As, Ps = _constant_sa(case["nx"], case["ny"], case["nz"])
        S = Solver().load(As, Ps)
        S.set_smoother(-1, case["kind"], case["degree"])
        S.set_coarse_sweeps(30)
        S.set_flexible("fcg1")
        b = _vec(seed, _n(case))
        s.update(S=S, b=b, x=torch.empty_like(b))
    elif what == "train":
        p = learn.Problem(_hierarchy(case, seed), nvec=case["m"], seed=seed)
        case = dict(case, degree=learn.DEGREE)
        s.update(p=p, betas=_weights(case, seed))
    elif what == "grad":
        S = Solver().load(*_csr(_hierarchy(case, seed)))
        r = _vec(seed, _n(case)).requires_grad_()
        betas = torch.from_numpy(_weights(case, seed)).requires_grad_()
        s.update(S=S, r=r, betas=betas, gz=_vec(seed + 1, _n(case)))
    else:
        S = Solver().load(*_csr(_hierarchy(case, seed)), prec=case["prec"])
        _set(S, case, seed)
        if what == "pcg":
            S.set_flexible(case["outer"])
        b = _vec(seed, _n(case))
        s.update(S=S, b=b, x=torch.empty_like(b))
        if what == "smooth":
            s.update(x0=_vec(seed + 1, _n(case)))
    return s


def _csr(H):
    return H.A, H.P


def run(s):
    case = s["case"]
    what = case["what"]
    if what == "smooth":
        x = s["x"] if case["zero"] else s["x"].copy_(s["x0"])
        s["S"].smooth(0, case["kind"], case["degree"], s["b"], x, x_is_zero=case["zero"])
        return x
    if what == "vcycle":
        s["S"].vcycle(s["b"], s["x"])
        return s["x"]
    if what in ("pcg", "sa_pcg"):
        it, rel = s["S"].pcg(s["b"], s["x"], rtol=1e-7 if what == "sa_pcg" else 1e-8)
        return dict(x=s["x"], iters=it, relres=rel)
    if what == "grad":
        s["r"].grad = s["betas"].grad = None
        z = VCycleFn.apply(s["r"], s["betas"], s["S"])
        z.backward(s["gz"])
        return dict(z=z, gr=s["r"].grad, gbetas=s["betas"].grad)
    if what == "train":
        loss, g = s["p"].loss_grad(s["betas"])
        return dict(loss=loss, g=g)
    if what == "mlp":
        net = s["net"]
        F, beta, acts = net.forward(s["feats"])
        net.backward_and_step(F, beta, acts, s["gbeta"], 2e-3)
        return dict(beta=beta, grads=net.grads, params=net.params, m=net.m, v=net.v)
    As, Ps, omegas = s["S"].sa_hierarchy(s["A"], s["levels"])
    out = dict(omegas=omegas)
    for l, (A, P) in enumerate(zip(As[1:], Ps)):
        for k, M in (("A", A), ("P", P)):
            out["%s%d" % (k, l)] = dict(ptr=M.indptr, col=M.indices, val=M.data)
    return out


def work(case):
    """Bytes and flops of one pass: each product of an iteration reads its
    matrix once and its vectors once (8/7 for the coarser levels)."""
    what = case["what"]
    if what == "mlp":
        B = case["batch"]
        return dict(bytes=4.0 * (7 * 4996 + B * (8 + 8 + 2 * 132)), flops=6.0 * 4864 * B)
    n = float(_n(case))
    k = case.get("degree", learn.DEGREE)
    v = dict(f64=8, f32=4, bf16=2)[case.get("prec", "f64")]
    x = 8 if v == 8 else 4
    prod = 7 * v * n + 2 * x * n          # one product on the finest level
    cyc = 8.0 / 7.0 * 2 * k               # products of one V-cycle, in finest-level products
    if what == "smooth":
        p = k - (1 if case["zero"] else 0)
        return dict(bytes=p * 7 * v * n + 16 * n, flops=14.0 * n * p)
    if what == "vcycle":
        return dict(bytes=cyc * 7 * v * n + 16 * n, flops=14.0 * n * cyc)
    if what == "pcg":
        it = round(1.25 * math.log2(n)) * (3 if case["problem"] == "aniso" else 1)
        return dict(bytes=it * (cyc * prod + 7 * 8 * n + 16 * n), flops=it * 14.0 * n * (cyc + 1))
    if what == "grad":
        return dict(bytes=2.5 * cyc * prod, flops=2.5 * cyc * 14.0 * n)
    if what == "train":
        # the matrices serve all m vectors of a product
        c = (learn.PRE_CYCLES + 2.5) * cyc + learn.PRE_CYCLES + 2
        return dict(bytes=c * (7 * v * n + 2 * x * n * case["m"]), flops=c * 14.0 * n * case["m"])
    if what == "sa_pcg":
        # operator complexity about 2.2, prolongators about 4.5 entries a row
        return dict(bytes=7 * (2.2 * 2 * k * prod + 2 * 12 * 4.5 * n + prod),
                    flops=7 * 14.0 * n * (2.2 * 2 * k + 2))
    # A in; about 4.5 entries a row of P and 8.4 of the coarse operators out
    return dict(bytes=(7 + 4.5 + 8.4) * 12 * n, flops=2.0 * n * (7 + 7 * 4.5 + 4.5 * 20))


# ---- the same results in 64-bit torch -----------------------------------------

class _Grid:
    """A 7-point operator on (..., nz, ny, nx) tensors."""

    def __init__(self, diag, cx, cy, cz):
        self.d, self.cx, self.cy, self.cz = diag, cx, cy, cz
        self.shape = tuple(diag.shape)

    def rounded(self, dtype):
        return _Grid(*(t.to(dtype).double() for t in (self.d, self.cx, self.cy, self.cz)))

    @functools.cached_property
    def minv(self):
        m = self.d.clone()
        for c, a in ((self.cx, 2), (self.cy, 1), (self.cz, 0)):
            k = c.shape[a]
            m.narrow(a, 0, k).add_(c.abs())
            m.narrow(a, 1, k).add_(c.abs())
        return 1.0 / m

    def mul(self, u):
        y = self.d * u
        for c, a in ((self.cx, -1), (self.cy, -2), (self.cz, -3)):
            k = c.shape[a]
            up, down = c * u.narrow(a, 1, k), c * u.narrow(a, 0, k)
            pad = [0, 0] * (-a - 1)
            y = y - torch.nn.functional.pad(up, pad + [0, 1])
            y = y - torch.nn.functional.pad(down, pad + [1, 0])
        return y

    def coarser(self):
        def ext(c, a):   # couplings between two blocks
            i = torch.arange(1, c.shape[a], 2, device=c.device)
            return _pairs(c.index_select(a, i), [x for x in (0, 1, 2) if x != a])

        d = _pairs(self.d, (0, 1, 2))
        for c, a in ((self.cx, 2), (self.cy, 1), (self.cz, 0)):
            i = torch.arange(0, c.shape[a], 2, device=c.device)
            inner = _pairs(c.index_select(a, i), [x for x in (0, 1, 2) if x != a])
            d.narrow(a, 0, inner.shape[a]).sub_(2 * inner)
        return _Grid(d, ext(self.cx, 2), ext(self.cy, 1), ext(self.cz, 0))

    @functools.cached_property
    def inverse(self):
        n = math.prod(self.shape)
        eye = torch.eye(n, dtype=torch.float64, device="cuda").view(n, *self.shape)
        return torch.linalg.inv(self.mul(eye).reshape(n, n))


def _pairs(t, axes):
    """Sums of consecutive pairs along the last-three axes `axes` (0, 1, 2)."""
    for a in axes:
        a = t.dim() - 3 + a
        if t.shape[a] % 2:
            pad = [0, 0] * (t.dim() - 1 - a) + [0, 1]
            t = torch.nn.functional.pad(t, pad)
        t = t.unflatten(a, (t.shape[a] // 2, 2)).sum(a + 1)
    return t


def _spread(t, shape):
    for a, s in zip((-3, -2, -1), shape):
        t = t.repeat_interleave(2, dim=a).narrow(a, 0, s)
    return t


def _smooth(mul, minv, b, x, kind, k, w=None):
    """x <- S(b, x) (x None: from zero)."""
    r = b if x is None else b - mul(x)
    if kind == "l1jacobi":
        for j in range(k):
            z = minv * r
            x = z if x is None else x + z
            r = b - mul(x) if j < k - 1 else r
        return x
    if kind == "cheb1_opt":
        theta, delta = 0.5 * (1.0 + ASTAR[k]), 0.5 * (1.0 - ASTAR[k])
        sigma = theta / delta
        rho = 1.0 / sigma
        z = minv * r / theta
        x = z if x is None else x + z
        for _ in range(1, k):
            r = r - mul(z)
            new = 1.0 / (2.0 * sigma - rho)
            z = new * rho * z + 2.0 * new / delta * (minv * r)
            x, rho = x + z, new
        return x
    beta = w if w is not None else BETA[k] if kind == "cheb4_opt" else [1.0] * k
    z = None
    for j in range(1, k + 1):
        y = (8 * j - 4) / (2 * j + 1) * (minv * r)
        z = y if z is None else y + (2 * j - 3) / (2 * j + 1) * z
        x = beta[j - 1] * z if x is None else x + beta[j - 1] * z
        r = r - mul(z) if j < k else r
    return x


class _Amg:
    """The V-cycle on a list of grids, coarsest last."""

    def __init__(self, case, seed, ws=None):
        st = _stencil(case, seed)
        g = _Grid(*(torch.from_numpy(np.ascontiguousarray(a)).cuda()
                    for a in (st.diag, st.cx, st.cy, st.cz)))
        self.A = g
        self.g = [g]
        for _ in _levels(case)[1:]:
            self.g.append(self.g[-1].coarser())
        self.coarse = self.g[-1].inverse
        if case.get("prec") == "bf16":
            self.g = [x.rounded(torch.bfloat16) for x in self.g]
        self.kind, self.k, self.ws = case.get("kind", "weights"), case.get("degree", 4), ws

    def one(self, l, b, x):
        g = self.g[l]
        return _smooth(g.mul, g.minv, b, x, self.kind, self.k, None if self.ws is None else self.ws[l])

    def cycle(self, b, l=0):
        g = self.g[l]
        if l == len(self.g) - 1:
            return (b.flatten(-3) @ self.coarse).view(b.shape)
        x = self.one(l, b, None)
        e = self.cycle(_pairs(b - g.mul(x), (0, 1, 2)), l + 1)
        return self.one(l, b, x + _spread(e, g.shape))


def _pcg(mul, M, b, rtol, outer):
    dot = lambda u, v: float((u * v).sum())  # noqa: E731
    x, r = torch.zeros_like(b), b.clone()
    b0 = math.sqrt(dot(b, b))
    z = M(r)
    p, rz = z.clone(), dot(r, z)
    for it in range(1, 1001):
        q = mul(p)
        alpha = rz / dot(p, q)
        x += alpha * p
        r = r - alpha * q
        rel = math.sqrt(dot(r, r)) / b0
        if rel <= rtol:
            break
        old, z = z, M(r)
        new = dot(r, z)
        beta = (new - (dot(r, old) if outer == "flexible" else 0.0)) / rz
        p, rz = z + beta * p, new
    return x, rel


class _Sa:
    """Smoothed aggregation on torch sparse matrices."""

    def __init__(self, A, levels):
        n = A.shape[0]
        self.A = [torch.sparse_csr_tensor(torch.from_numpy(A.indptr).cuda(),
                                          torch.from_numpy(A.indices).cuda(),
                                          torch.from_numpy(A.data).cuda(), (n, n))]
        self.P, self.omega = [], []
        for agg, nc, _ in levels:
            A, n = self.A[-1], self.A[-1].shape[0]
            agg = torch.from_numpy(agg).cuda().long()
            rows = _row_ids(A)
            val, col = A.values(), A.col_indices().long()
            d = torch.zeros(n, dtype=torch.float64, device="cuda")
            d.index_add_(0, rows, torch.where(rows == col, val, 0.0))
            s = torch.zeros_like(d).index_add_(0, rows, val.abs())
            om = 4.0 / (3.0 * float((s / d).max()))
            # (I - omega D^-1 A) P_hat: columns mapped to their aggregates
            v = -om * val / d[rows] + torch.where(rows == col, 1.0, 0.0)
            P = _csr_of(rows, agg[col], v, (n, nc))
            self.P.append(P)
            self.omega.append(om)
            AP = torch.sparse.mm(A, P)
            T = _csr_of(P.col_indices().long(), _row_ids(P), P.values(), (nc, n))
            C = torch.sparse.mm(T, AP)
            self.A.append(_csr_of(_row_ids(C), C.col_indices().long(), C.values(), (nc, nc)))

    def solver(self, kind, k, sweeps):
        mats = [(A, self.P[l] if l < len(self.P) else None) for l, A in enumerate(self.A)]
        rs = [_csr_of(P.col_indices().long(), _row_ids(P), P.values(), P.shape[::-1])
              for P in self.P]
        minv = [1.0 / torch.zeros(A.shape[0], dtype=torch.float64, device="cuda").index_add_(
            0, _row_ids(A), A.values().abs()) for A in self.A]

        def cycle(b, l=0):
            A, P = mats[l]
            mul = lambda u: A @ u  # noqa: E731
            if P is None:
                return _smooth(mul, minv[l], b, None, "l1jacobi", sweeps)
            x = _smooth(mul, minv[l], b, None, kind, k)
            x = x + P @ cycle(rs[l] @ (b - A @ x), l + 1)
            return _smooth(mul, minv[l], b, x, kind, k)
        return cycle


def _row_ids(A):
    p = A.crow_indices().long()
    return torch.repeat_interleave(torch.arange(A.shape[0], device="cuda"), p[1:] - p[:-1])


def _csr_of(rows, cols, val, shape):
    return torch.sparse_coo_tensor(torch.stack((rows, cols)), val, shape).coalesce().to_sparse_csr()


def exact(case, seed):
    what = case["what"]
    if what == "mlp":
        return _exact_mlp(case, seed)
    if what == "sa_setup":
        s = prepare(case, seed)
        sa = _Sa(s["A"], s["levels"])
        out = dict(omegas=sa.omega)
        for l in range(len(sa.P)):
            for k, M in (("A", sa.A[l + 1]), ("P", sa.P[l])):
                out["%s%d" % (k, l)] = dict(ptr=None, col=None, val=M.values())
        return out
    if what == "sa_pcg":
        st = pr.poisson(case["nx"], case["ny"], case["nz"])
        sa = _Sa(pr.to_csr(st), pr.geometric_aggregates(st.shape, COARSE_MAX))
        x, rel = _pcg(lambda u: sa.A[0] @ u, sa.solver(case["kind"], case["degree"], 30),
                      _vec(seed, _n(case)), 1e-7, "cg")
        return dict(x=x, iters=None, relres=rel)
    shape = (case["nz"], case["ny"], case["nx"])
    if what == "train":
        return _exact_train(dict(case, degree=learn.DEGREE), seed)
    if what == "grad":
        amg = _Amg(case, seed, torch.from_numpy(_weights(case, seed)).cuda().requires_grad_())
        r = _vec(seed, _n(case)).view(shape).requires_grad_()
        z = amg.cycle(r)
        z.backward(_vec(seed + 1, _n(case)).view(shape))
        return dict(z=z.detach().flatten(), gr=r.grad.flatten(), gbetas=amg.ws.grad)
    amg = _Amg(case, seed, _weights(case, seed) if case["kind"] == "weights" else None)
    b = _vec(seed, _n(case)).view(shape)
    if what == "smooth":
        return amg.one(0, b, None if case["zero"] else _vec(seed + 1, _n(case)).view(shape)).flatten()
    if what == "vcycle":
        return amg.cycle(b).flatten()
    x, rel = _pcg(amg.A.mul, amg.cycle, b, 1e-8, case["outer"])
    # with 16- or 32-bit values the last residual is another one
    return dict(x=x.flatten(), iters=None, relres=rel if case["prec"] == "f64" else None)


def _exact_train(case, seed):
    """Mean A-norm reduction of one V-cycle after the pre-cycles, and its gradient."""
    w = np.stack([learn.make_safe(b, np.asarray(BETA[4]))[0] for b in _weights(case, seed)])
    amg = _Amg(case, seed, torch.from_numpy(w).cuda())
    E = torch.from_numpy(pr.vec_normal(_n(case), seed=seed, count=case["m"])).cuda()
    loss, g = 0.0, 0.0
    for e in E.view(-1, case["nz"], case["ny"], case["nx"]).split(4):
        amg.ws = amg.ws.detach()
        for _ in range(learn.PRE_CYCLES):
            e = e - amg.cycle(amg.A.mul(e))
        amg.ws.requires_grad_()
        e1 = e - amg.cycle(amg.A.mul(e))
        norm = lambda u: (u * amg.A.mul(u)).sum((-3, -2, -1))  # noqa: E731
        part = (norm(e1) / norm(e)).sum() / case["m"]
        g = g + torch.autograd.grad(part, amg.ws)[0]
        loss = loss + float(part.detach())
    return dict(loss=loss, g=g)


def _exact_mlp(case, seed):
    net, feats, gbeta = _mlp_inputs(case, seed)
    th = net.params.double().requires_grad_()
    f = torch.from_numpy(feats).cuda().double()
    h = torch.relu(f @ th[:512].view(64, 8).T + th[512:576])
    h = torch.relu(h @ th[576:4672].view(64, 64).T + th[4672:4736])
    o = h @ th[4736:4992].view(4, 64).T + th[4992:]
    beta = torch.tensor(BETA[4], dtype=torch.float64, device="cuda") * torch.exp(2 * torch.tanh(o / 2))
    beta.backward(torch.from_numpy(gbeta).cuda().double())
    g = th.grad
    m, v = 0.1 * g, 0.001 * g * g
    step = 2e-3 * (m / 0.1) / (torch.sqrt(v / 0.001) + 1e-8)
    return dict(beta=beta.detach().flatten(), grads=g, params=th.detach() - step, m=m, v=v)

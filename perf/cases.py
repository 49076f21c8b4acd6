"""What is timed: calls a user of this package makes, from one operator application on the smallest
lattice to a batched solve.

Every case is a plain dict.  `prepare` makes what the caller has in hand before the call (a context with
its gauge field, rational function and, where the case has any, deflation data; the fields on the GPU),
`run` makes the call, `exact` gives the same numbers in 64 bits from plain torch and numpy.

Sizes are those of the package's own workloads (4^4, 6^4, 8^4, 10^4, 24^4; s = 16 or 20 poles, k = 30 or
40, 1 or 12 right-hand sides, random SU(3) links of spread 0.5 or 0.7, mu = 0.2, 0.3, 0.5), plus ragged
lattices.  Solves run at the context's default tolerance, 1e-10."""
import math

import numpy as np
import torch

import paper_0910_2927_gb300 as sgn
from paper_0910_2927_gb300.autograd import SignApply

LINKS = {"fp32": sgn.LINKS_FP32, "fp16": sgn.LINKS_FP16, "bf16": sgn.LINKS_BF16}
MASS = -1.6  # the contexts' default kernel mass


def _case(name, what, dims, nrhs=1, mu=0.3, spread=0.7, **more):
    c = {"what": what, "lx": dims[0], "ly": dims[1], "lz": dims[2], "lt": dims[3], "nrhs": nrhs, "mu": mu,
         "spread": spread, **more}
    return {"name": name, **c} if name else c


def _hw(name, dims, nrhs, arith="f64", links="fp32", packed=False, adjoint=False, **more):
    return _case(name, "hw", dims, nrhs, arith=arith, links=links, packed=packed, adjoint=adjoint, **more)


def _solve(name, dims, nrhs, form="f64", links="fp32", method="fom", m=0, s=20, k=40, adjoint=False, source="gauss",
           **more):
    return _case(name, "solve", dims, nrhs, form=form, links=links, method=method, m=m, s=s, k=k, adjoint=adjoint,
                 source=source, **more)


def listed():
    return [
        # one operator application on the smallest workload lattice: a call's latency
        _hw("hw 4^4 f64 x1", (4, 4, 4, 4), 1, spread=0.5),
        # FP64 operator on a propagator's twelve fields, backward direction (H_W(mu)^dag)
        _hw("hw 10^4 f64 x12 adjoint", (10, 10, 10, 10), 12, adjoint=True),
        # the bandwidth case: FP32 operator, twelve packed fields far larger than L2
        _hw("hw 24^4 f32 x12 packed", (24, 24, 24, 24), 12, "f32", packed=True, mu=0.2),
        # natural-order fields, 16-bit links, odd extents and an odd number of fields
        _hw("hw 15x13x18x22 f32 x5 fp16", (15, 13, 18, 22), 5, "f32", links="fp16"),
        # float-float operator: residuals to 64-bit accuracy without the FP64 units
        _hw("hw 16^4 ff x4", (16, 16, 16, 16), 4, "ff", mu=0.2),
        # projection and Gram-Schmidt coefficients against a deflation-sized basis
        _case("inner products 16^4 30x12", "dots", (16, 16, 16, 16), 12, basis=30),
        # the smallest solve, plain FP64 form, deflated: one column on 4^4
        _solve("solve 4^4 f64 x1 m8", (4, 4, 4, 4), 1, m=8, s=16, k=30, spread=0.5),
        # one Gaussian source on 6^4, mixed form, deflated
        _solve("solve 6^4 mixed x1 m8", (6, 6, 6, 6), 1, "mixed", m=8),
        # a propagator: twelve point sources in one batched solve on 10^4, mixed form
        _solve("solve 10^4 mixed x12", (10, 10, 10, 10), 12, "mixed", source="point"),
        # plain FP64 form on a ragged lattice, three columns
        _solve("solve 7x6x9x8 f64 x3", (7, 6, 9, 8), 3),
        # training step on 6^4: forward and backward through the autograd function, d/db and d/dmu
        _case("grad 6^4 f64 x1", "grad", (6, 6, 6, 6), 1, mu=0.5, s=20, k=40),
        # the direct projection of eq. (6.3) the method is compared with
        _case("direct 8^4 k100 x2", "direct", (8, 8, 8, 8), 2, k=100),
    ]


def draw(rng):
    def extents(lo, hi, most):
        while True:
            d = tuple(int(round(math.exp(rng.uniform(math.log(lo), math.log(hi))))) for _ in range(4))
            if math.prod(d) <= most:
                return d

    what = rng.choice(["hw", "hw", "hw", "solve", "solve", "solve", "dots", "grad", "direct"])
    mu = round(rng.uniform(0.0, 0.35), 3)
    spread = round(rng.uniform(0.5, 0.7), 3)
    nrhs = int(round(math.exp(rng.uniform(0.0, math.log(12.4)))))
    if what == "hw":
        arith = rng.choice(["f64", "f32", "f32", "ff"])
        return _hw(None, extents(3, 24.4, 16 ** 4 if arith != "f32" else 24 ** 4), nrhs, arith,
                   rng.choice(["fp32", "fp32", "fp16", "bf16"]) if arith == "f32" else "fp32",
                   rng.random() < 0.4, rng.random() < 0.3, mu=mu, spread=spread)
    if what == "solve":
        form = rng.choice(["f64", "mixed", "mixed"])
        most = 10 ** 4 if form == "mixed" else 12000 // nrhs  # FP64 costs more: smaller in all
        links = rng.choice(["fp32", "fp32", "fp16"]) if form == "mixed" else "fp32"
        method = rng.choice(["fom", "fom", "gmres"]) if form == "f64" else "fom"
        return _solve(None, extents(4, 10.4, most), nrhs, form, links, method, 0, rng.randint(12, 20),
                      rng.randint(30, 40), rng.random() < 0.3, rng.choice(["gauss", "point"]), mu=mu, spread=spread)
    if what == "dots":
        return _case(None, "dots", extents(3, 16.4, 16 ** 4), nrhs, mu=mu, spread=spread, basis=rng.randint(1, 64))
    if what == "grad":
        return _case(None, "grad", extents(4, 7.4, 6 ** 4), min(nrhs, 2), mu=mu, spread=spread, s=rng.randint(12, 20),
                     k=rng.randint(30, 40))
    return _case(None, "direct", extents(4, 8.4, 8 ** 4), min(nrhs, 2), mu=mu, spread=spread, k=rng.randint(40, 100))


# ------------------------------------------------------------------ inputs --

def _dims(c):
    return c["lx"], c["ly"], c["lz"], c["lt"]


def _vol(c):
    return c["lx"] * c["ly"] * c["lz"] * c["lt"]


def _gaussian(g, *shape):
    z = torch.randn(*shape, 2, dtype=torch.float64, device="cuda", generator=g)
    return torch.view_as_complex(z) / math.sqrt(2.0)


def _links(c, g):
    """exp(i spread sum_a g_a lambda_a / 2), g_a ~ N(0, 1): (V, 4, 3, 3), random SU(3) links."""
    z = torch.randn(_vol(c) * 4, 8, dtype=torch.float64, device="cuda", generator=g)
    h = torch.zeros(z.shape[0], 3, 3, dtype=torch.complex128, device="cuda")
    for a, (i, j) in ((0, (0, 1)), (3, (0, 2)), (5, (1, 2))):
        h[:, i, j] = torch.complex(z[:, a], -z[:, a + 1])
        h[:, j, i] = torch.complex(z[:, a], z[:, a + 1])
    r3 = 1.0 / math.sqrt(3.0)
    h[:, 0, 0] = z[:, 2] + z[:, 7] * r3
    h[:, 1, 1] = -z[:, 2] + z[:, 7] * r3
    h[:, 2, 2] = -2.0 * z[:, 7] * r3
    x = h * (0.5j * c["spread"] / 16.0)  # the exponential by scaling and squaring
    u = torch.eye(3, dtype=torch.complex128, device="cuda").expand_as(x)
    for q in range(14, 0, -1):
        u = torch.eye(3, dtype=torch.complex128, device="cuda") + (x @ u) / q
    for _ in range(4):
        u = u @ u
    return u.reshape(_vol(c), 4, 3, 3).contiguous()


def _inputs(c, seed):
    g = torch.Generator(device="cuda").manual_seed(int(seed))
    n, nrhs = 12 * _vol(c), c["nrhs"]
    if c["what"] == "dots":
        return {"V": _gaussian(g, c["basis"], n), "w": _gaussian(g, nrhs, n)}
    d = {"U": _links(c, g)}
    if c.get("source") == "point":  # unit vectors at site 0: column 3 spin + colour
        d["b"] = torch.zeros(nrhs, n, dtype=torch.complex128, device="cuda")
        for r in range(nrhs):
            d["b"][r, r % 12] = 1.0
    else:
        d["b"] = _gaussian(g, nrhs, n)
    if c["what"] == "hw" and c["arith"] == "f32":
        d["b"] = d["b"].to(torch.complex64)
    if c["what"] == "grad":
        d["g"] = _gaussian(g, nrhs, n)
    return d


def _rational(c):
    """Poles scaled to the spectrum: c = 1/sqrt(a b), a near the smallest |lambda| these links give, b a bound."""
    return sgn.kenney_laub(c["s"], 1.0 / math.sqrt(0.2 * _bound(c)))


def _bound(c):
    return abs(4.0 + MASS) + 3.0 * math.sqrt(2.0) + math.sqrt(2.0 * math.cosh(2.0 * c["mu"]))


# -------------------------------------------------------------- the calls --

def prepare(case, seed):
    c = case
    d = _inputs(c, seed)
    ctx = sgn.SignContext(_dims(c), mu=c["mu"])
    st = {"case": dict(c), "ctx": ctx, **d}
    if c["what"] == "dots":
        return st
    ctx.load_gauge(st.pop("U"))
    if c["what"] == "hw":
        if c["arith"] == "f32":
            ctx.set_precision(sgn.PREC_MIXED, 1e-8, LINKS[c["links"]])
        if c["packed"]:
            st["b"] = ctx.pack(st["b"], sgn.PREC_MIXED if c["arith"] == "f32" else sgn.PREC_FP64)
    if c["what"] in ("solve", "grad"):
        ctx.set_rational(*_rational(c))
        ctx.set_restart(k=c["k"], tol=1e-10 if c["what"] == "solve" else 1e-12)
    if c["what"] == "solve":
        if c["m"]:
            ctx.build_deflation(c["m"], extra=4, eig_tol=1e-11)
        ctx.set_method(sgn.METHOD_GMRES if c["method"] == "gmres" else sgn.METHOD_FOM)
        if c["form"] == "mixed":
            ctx.set_precision(sgn.PREC_MIXED, 1e-8, LINKS[c["links"]])
    return st


def run(state):
    c, ctx = state["case"], state["ctx"]
    if c["what"] == "hw":
        return ctx.hw(state["b"], precision=sgn.PREC_MIXED if c["arith"] == "f32" else sgn.PREC_FP64,
                      adjoint=c["adjoint"], packed=c["packed"], float_float=c["arith"] == "ff")
    if c["what"] == "dots":
        return ctx.inner_products(state["V"], state["w"])
    if c["what"] == "solve":
        return ctx.apply(state["b"], adjoint=c["adjoint"])[0]
    if c["what"] == "direct":
        return ctx.apply_direct(state["b"], c["k"])[0]
    b = state["b"].clone().requires_grad_(True)
    mu = torch.tensor(c["mu"], dtype=torch.float64, requires_grad=True)
    x = SignApply.apply(b, mu, ctx)
    x.backward(state["g"])
    return {"x": x.detach(), "b": b.grad, "mu": mu.grad}


def work(case):
    c, v, nrhs = case, _vol(case), case["nrhs"]
    n = 12 * v
    field, links, hop = 16.0 * n, 16.0 * 36 * v, 1368.0 * v  # complex128 bytes; flops of one H_W on one field
    if c["what"] == "dots":
        return {"bytes": field * (c["basis"] + nrhs), "flops": 8.0 * n * c["basis"] * nrhs}
    if c["what"] == "hw":
        if c["arith"] == "f32":
            field, links = field / 2, links / (2 if c["links"] == "fp32" else 4)
        return {"bytes": 2 * field * nrhs + links, "flops": hop * nrhs}
    if c["what"] == "direct":  # k applications of A; every basis vector enters two Gram-Schmidt passes
        return {"bytes": 2 * field * nrhs + links, "flops": nrhs * (c["k"] * hop + 8.0 * n * c["k"] * (c["k"] + 2))}
    # a Krylov space of A^2 of the dimension the slowest shift needs by the Chebyshev estimate
    tol, kappa = 1e-10 if c["what"] == "solve" else 1e-12, (_bound(c) / 0.2) ** 2
    steps = math.ceil(math.sqrt(kappa) * math.log(2.0 / tol) / 4.0)
    solves = 1 if c["what"] == "solve" else 4  # forward, adjoint, and the per-shift pair of the mu-derivative
    return {"bytes": (2 * solves) * field * nrhs + links, "flops": solves * nrhs * 2.0 * steps * hop}


# ------------------------------------------------ the same in 64 bits --

_SIGMA = (((0, 1), (1, 0)), ((0, -1j), (1j, 0)), ((1, 0), (0, -1)))


def _gammas():
    out = []
    for s in _SIGMA:
        m = torch.zeros(4, 4, dtype=torch.complex128)
        m[:2, 2:] = -1j * torch.tensor(s, dtype=torch.complex128)
        m[2:, :2] = 1j * torch.tensor(s, dtype=torch.complex128)
        out.append(m.cuda())
    m = torch.zeros(4, 4, dtype=torch.complex128)
    m[:2, 2:] = m[2:, :2] = torch.eye(2)
    return out + [m.cuda()]


class _Operator:
    """gamma5 D_W(mu) on fields (..., n); antiperiodic in t; dmu: its derivative with respect to mu."""

    def __init__(self, c, U, mu):
        self.shape = (c["lt"], c["lz"], c["ly"], c["lx"])
        self.U = U.reshape(*self.shape, 4, 3, 3)
        self.mu, self.gamma = mu, _gammas()
        self.g5 = torch.tensor([1.0, 1.0, -1.0, -1.0], dtype=torch.float64, device="cuda")[:, None]

    def __call__(self, psi, dmu=False):
        f = psi.reshape(-1, *self.shape, 4, 3)
        out = torch.zeros_like(f) if dmu else (4.0 + MASS) * f
        for nu in (3,) if dmu else range(4):
            ax = 4 - nu
            u = self.U[..., nu, :, :]
            fw, bw = (math.exp(self.mu), math.exp(-self.mu)) if nu == 3 else (1.0, 1.0)
            up = torch.roll(f, -1, ax)
            lo = torch.roll(torch.einsum("tzyxba,rtzyxsb->rtzyxsa", u.conj(), f), 1, ax)
            if nu == 3:
                up[:, -1] *= -1.0
                lo[:, 0] *= -1.0
            up = torch.einsum("tzyxab,rtzyxsb->rtzyxsa", u, up)
            out -= 0.5 * fw * (up - torch.einsum("sp,rtzyxpa->rtzyxsa", self.gamma[nu], up))
            back = 0.5 * bw * (lo + torch.einsum("sp,rtzyxpa->rtzyxsa", self.gamma[nu], lo))
            out = out + back if dmu else out - back
        return (out * self.g5).reshape(psi.shape)


def _arnoldi(op, r, most, coefficients):
    """Orthonormal basis of one column's Krylov space of `op` from r until the coefficients settle:
    (basis, coefficients): sum_j coefficients_j basis_j is the function's value."""
    V = torch.empty(most + 1, r.numel(), dtype=torch.complex128, device="cuda")
    H = np.zeros((most + 1, most), dtype=np.complex128)
    beta = float(torch.linalg.vector_norm(r))
    V[0] = r / beta
    k = 0
    while k < most:
        w = op(V[k])
        h = torch.zeros(k + 1, dtype=torch.complex128, device="cuda")
        for _ in range(2):
            p = (V[:k + 1].conj() @ w)
            w = w - p @ V[:k + 1]
            h += p
        H[:k + 1, k] = h.cpu().numpy()
        H[k + 1, k] = float(torch.linalg.vector_norm(w))
        k += 1
        if abs(H[k, k - 1]) < 1e-13 * abs(H[:k, :k]).max():
            break
        V[k] = w / float(H[k, k - 1].real)
        if k % 40 == 0:
            y = coefficients(H[:k, :k])
            if np.linalg.norm(y[..., -8:]) < 1e-13 * np.linalg.norm(y):
                break
    return V[:k], beta * coefficients(H[:k, :k])


def _shifted(sigma):
    def y(H):
        e = np.zeros(H.shape[0], dtype=np.complex128)
        e[0] = 1.0
        return np.stack([np.linalg.solve(H - s * np.eye(H.shape[0]), e) for s in sigma])
    return y


def _critical(A, m):
    """The m eigenvalues of smallest modulus of a dense A, their right vectors as rows R and their left vectors
    as rows L with conj(L) R^T = 1: by Arnoldi on the inverse, whose largest eigenvalues they are."""
    def largest(inv):
        g = torch.Generator(device="cuda").manual_seed(1)
        last = {}

        def keep(H):
            last["H"] = H
            return np.ones(H.shape[0])  # never settles: the whole space asked for
        V, _ = _arnoldi(lambda v: inv @ v, _gaussian(g, inv.shape[0]), 360, keep)
        theta, s = np.linalg.eig(last["H"])
        at = np.argsort(-abs(theta))[:m]
        return theta[at], torch.from_numpy(np.ascontiguousarray(s[:, at].T)).cuda() @ V
    inv = torch.linalg.inv(A)
    theta, R = largest(inv)
    _, L = largest(inv.conj().T.contiguous())
    return 1.0 / theta, R, torch.linalg.inv(R @ L.conj().T).conj().T @ L


def exact(case, seed):
    c = case
    d = _inputs(c, seed)
    if c["what"] == "dots":
        return (d["w"] @ d["V"].conj().T).cpu().numpy()
    U, b = d["U"], d["b"].to(torch.complex128)
    if c["what"] == "hw":
        if c["arith"] == "f32":  # the operator on the links as stored
            short = {"fp32": torch.float32, "fp16": torch.float16, "bf16": torch.bfloat16}[c["links"]]
            U = torch.view_as_complex(torch.view_as_real(U).float().to(short).double())
        out = torch.cat([_Operator(c, U, -c["mu"] if c["adjoint"] else c["mu"])(v[None]) for v in b])
        if c["packed"]:
            out = out.reshape(c["nrhs"], -1, 6, 2).transpose(1, 2).reshape(c["nrhs"], -1)
        return out.contiguous()
    if c["what"] == "direct":
        A = _Operator(c, U, c["mu"])

        def sign_first(H):
            lam, X = np.linalg.eig(H)
            e = np.zeros(H.shape[0], dtype=np.complex128)
            e[0] = 1.0
            return X @ (np.sign(lam.real) * np.linalg.solve(X, e)) + 0.0
        out = []
        for v in b:  # exactly k steps, converged or not: that is the method
            V, y = _arnoldi(A, v, c["k"], lambda H: sign_first(H) if H.shape[0] == c["k"] else np.ones(H.shape[0]))
            out.append(torch.from_numpy(y).cuda() @ V)
        return torch.stack(out)
    sigma, omega = _rational(c)
    w = torch.from_numpy(omega).to(torch.complex128).cuda()

    def iterates(mu, v):  # (A^2 - sigma_i)^-1 v
        A = _Operator(c, U, mu)
        V, y = _arnoldi(lambda q: A(A(q)), v, 1200, _shifted(sigma))
        return torch.from_numpy(y).cuda() @ V

    if c["what"] == "solve":
        mu = -c["mu"] if c["adjoint"] else c["mu"]
        A = _Operator(c, U, mu)
        x = torch.stack([w @ iterates(mu, A(v)) for v in b])
        if c["m"]:  # the deflated eigenvalues get their exact sign in place of the rational function's value
            n = 12 * _vol(c)
            if n > 3200:
                return None
            lam, R, L = _critical(A(torch.eye(n, dtype=torch.complex128, device="cuda")).T, c["m"])
            g = (omega[None] * lam[:, None] / (lam[:, None] ** 2 - sigma[None])).sum(1)
            x = x + (torch.from_numpy(np.sign(lam.real) - g).cuda() * (b @ L.conj().T)) @ R
        return x
    A, B = _Operator(c, U, c["mu"]), _Operator(c, U, -c["mu"])
    x, gb, gmu = [], [], 0.0
    for v, q in zip(b, d["g"]):
        xi, zi = iterates(c["mu"], A(v)), iterates(-c["mu"], q)
        x.append(w @ xi)
        gb.append(w @ torch.stack([B(z) for z in zi]))
        for i in range(c["s"]):
            t = A(v, True) - A(A(xi[i]), True) - A(A(xi[i], True))
            gmu += float((omega[i] * torch.vdot(zi[i], t)).real)
    return {"x": torch.stack(x), "b": torch.stack(gb), "mu": torch.tensor(gmu, dtype=torch.float64)}

"""The work that users have this library do, as calls of its public Python
entry points: what is timed and compared when a kernel changes.

Kinds of a case ("kind"):
  apply     Context.apply: D, D^H or A = D^H D on m fields in one storage
            precision: operator applications of a caller's own solver or
            measurement code.
  solve     Context.solve: (sigma_j + A) X_j = B for m right-hand sides and
            s shifts, every true residual below tol.
  schur     the same with the even-odd operator on odd-site half fields
            (Context.set_operator("schur")).
  grad      DSBCGSolve forward and backward: the solutions and the gradients
            of a loss of them, the incoming gradient one block per shift.
  rational  one molecular-dynamics step of rational HMC: new links
            (Context.update_gauge), Y = r(A) B (DSBCGRational forward) and its
            backward to B, the shifts and the links.
  force     Context.force: the gauge-link gradient from solutions and adjoint
            solutions that the caller holds.

Lattices, kappa, link smoothness eps, numbers of right-hand sides and shifts,
shift ranges and tolerances are those of synth.WORKLOADS and of the tests, and
sizes between them.  Links are exp(i eps H) with H a Gaussian traceless
hermitian matrix, put back onto SU(3), as in synth.su3_links; everything is
drawn on the GPU from the seed.
"""
import math

import torch

from paper_1205_0359_gb300 import dsbcg

LATTICE_MAX = 24 * 24 * 24 * 48        # sites of the largest lattice here
STORAGES = ("fp64", "fp32", "bf16", "fp16", "df32")


def _case(kind, lx, ly, lz, lt, m, s, storage, **kw):
    c = dict(kind=kind, lx=lx, ly=ly, lz=lz, lt=lt, m=m, s=s, storage=storage, op="A", kappa=0.125, eps=0.5,
             rhs="gaussian", lo=1e-4, hi=1.0, tol=1e-8, dependent=False)
    c.update(kw)
    return c


def listed():
    return [
        # the smallest call: one operator application on a test lattice, where launches and allocations count
        _case("apply", 4, 4, 4, 4, 4, 0, "fp64", name="apply_fp64_4x4x4x4", kappa=0.12, eps=0.3),
        # operator applications at the library's headline size, in the two storages that most callers use
        _case("apply", 16, 16, 16, 32, 12, 0, "fp64", name="apply_fp64_16x16x16x32"),
        _case("apply", 16, 16, 16, 32, 12, 0, "fp32", name="apply_fp32_16x16x16x32"),
        # one D^H in 16-bit storage on the lattice of the storage-precision ladder
        _case("apply", 24, 24, 24, 48, 8, 0, "bf16", name="apply_bf16_24x24x24x48", op="Ddag", kappa=0.13, eps=0.6),
        # the small FP64 solve with a dependent right-hand side (b_4 = b_1 + b_2), as in debugging and validation runs
        _case("solve", 4, 4, 4, 4, 4, 4, "fp64", name="solve_fp64_4x4x4x4", kappa=0.12, eps=0.3, lo=1e-3, tol=1e-10,
              dependent=True),
        # FP64 storage at the size and shifts of the paper's algorithm comparison
        _case("solve", 16, 16, 16, 16, 4, 7, "fp64", name="solve_fp64_16x16x16x16", lo=1e-6, hi=1e-1),
        # the headline: mixed precision, Z2 noise, the shifts of a partial-fraction expansion
        _case("solve", 16, 16, 16, 32, 12, 12, "fp32", name="solve_fp32_16x16x16x32", rhs="z2", hi=10.0),
        # the largest: mixed precision on the ladder's lattice
        _case("solve", 24, 24, 24, 48, 8, 8, "fp32", name="solve_fp32_24x24x24x48", kappa=0.13, eps=0.6),
        # the even-odd operator, as a production code would precondition
        _case("schur", 12, 12, 12, 24, 6, 10, "fp32", name="schur_fp32_12x12x12x24", hi=10.0),
        # gradients through the solve on a lattice of odd extents and a block width off the kernels' buckets
        _case("grad", 7, 9, 10, 13, 5, 3, "fp32", name="grad_fp32_7x9x10x13", lo=1e-2),
        # a rational-HMC step on a small production lattice, two pseudofermions
        _case("rational", 8, 8, 8, 16, 2, 8, "fp32", name="rational_fp32_8x8x8x16"),
        # the fermion force at the size at which the benchmark times it
        _case("force", 16, 16, 16, 32, 8, 8, "fp32", name="force_fp32_16x16x16x32"),
    ]


def _dims(rng, vol, even, least=2):
    """Four extents >= least whose product is near vol (ragged unless even)."""
    want = vol ** 0.25
    d = [max(least, int(round(want * math.exp(rng.uniform(-0.35, 0.35))))) for _ in range(3)]
    d.append(max(least, int(round(vol / (d[0] * d[1] * d[2])))))
    return [x + (x & 1) for x in d] if even else d


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    kind = rng.choice(("apply", "apply", "solve", "solve", "schur", "grad", "rational", "force"))
    kappa, eps = round(rng.uniform(0.11, 0.13), 4), round(rng.uniform(0.3, 0.6), 3)
    lo = 10.0 ** round(rng.uniform(-4, -2), 2)
    hi = 10.0 ** round(rng.uniform(-1, 1), 2)
    base = dict(kappa=kappa, eps=eps, lo=lo, hi=hi, rhs=rng.choice(("gaussian", "z2")))
    if kind == "apply":
        d = _dims(rng, _log(rng, 64, LATTICE_MAX / 2), False)
        return _case(kind, *d, rng.randint(1, 16), 0, rng.choice(STORAGES), op=rng.choice(("D", "Ddag", "A")), **base)
    if kind == "force":
        d = _dims(rng, _log(rng, 128, 100000), False)
        return _case(kind, *d, rng.randint(1, 8), rng.randint(1, 8), rng.choice(("fp64", "fp32")), **base)
    storage = rng.choice(("fp32", "fp32", "fp64"))
    # FP64 storage is for small lattices and narrow blocks; reduced storage goes up to the headline's size
    small = storage == "fp64" or kind in ("grad", "rational")
    d = _dims(rng, _log(rng, 256, 16000 if small else 100000), kind == "schur", 4)
    m, s = rng.randint(1, 6 if small else 12), rng.randint(1, 6 if small else 12)
    tol = 1e-10 if storage == "fp64" else 1e-8
    return _case(kind, *d, m, s, storage, tol=tol, dependent=rng.random() < 0.25, **base)


# ---------------------------------------------------------------- inputs --
def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return g


def _gauss(shape, g):
    """Complex Gaussian entries (g + i g') / sqrt(2)."""
    r = torch.randn(tuple(shape) + (2,), dtype=torch.float64, device="cuda", generator=g)
    return torch.view_as_complex(r) / math.sqrt(2.0)


def _links(c, g):
    """exp(i eps H) for every site and direction, rows made orthonormal and the third one the conjugate cross
    product of the others: [Lt][Lz][Ly][Lx][4][3][3]."""
    a = _gauss((c["lt"], c["lz"], c["ly"], c["lx"], 4, 3, 3), g)
    h = 0.5 * (a + a.mH)
    tr = torch.diagonal(h, dim1=-2, dim2=-1).sum(-1).real / 3.0
    h = 1j * c["eps"] * (h - tr[..., None, None] * torch.eye(3, dtype=h.dtype, device=h.device))
    u = torch.eye(3, dtype=h.dtype, device=h.device).expand_as(h).clone()
    t = u
    for k in range(1, 18):               # |eps H| is a few at most, and the rows are orthonormalised below
        t = (t.unsqueeze(-1) * h.unsqueeze(-3)).sum(-2) / k
        u = u + t
    r1 = u[..., 0, :] / torch.linalg.vector_norm(u[..., 0, :], dim=-1, keepdim=True)
    r2 = u[..., 1, :]
    r2 = r2 - (r1.conj() * r2).sum(-1, keepdim=True) * r1
    r2 = r2 / torch.linalg.vector_norm(r2, dim=-1, keepdim=True)
    r3 = torch.linalg.cross(r1, r2).conj()
    return torch.stack([r1, r2, r3], dim=-2).contiguous()


def _volume(c):
    return c["lx"] * c["ly"] * c["lz"] * c["lt"]


def _n(c):
    return (6 if c["kind"] == "schur" else 12) * _volume(c)


def _rhs(c, g):
    shape = (c["m"], _n(c))
    if c["rhs"] == "z2":
        r = torch.randint(0, 2, shape + (2,), device="cuda", generator=g).to(torch.float64) * 2 - 1
        b = torch.view_as_complex(r) / math.sqrt(2.0)
    else:
        b = _gauss(shape, g)
    if c["dependent"] and c["m"] >= 3:
        b[-1] = b[0] + b[1]
    return b


def _shifts(c):
    s, lo, hi = c["s"], c["lo"], c["hi"]
    if s == 1:
        return torch.tensor([lo], dtype=torch.float64)
    return 10.0 ** torch.linspace(math.log10(lo), math.log10(hi), s, dtype=torch.float64)


def _weights(c):
    return torch.linspace(0.1, 0.5, c["s"], dtype=torch.float64)


ALPHA0 = 0.25                             # the constant term of the rational function


def _draw_inputs(c, seed):
    """The case's inputs in a fixed order of draws, so that exact() has the same ones."""
    g = _gen(seed)
    d = dict(U=_links(c, g))
    if c["kind"] == "apply":
        d["B"] = _gauss((c["m"], _n(c)), g)
    elif c["kind"] == "force":
        d["X"] = _gauss((c["s"], c["m"], _n(c)), g)
        d["L"] = _gauss((c["s"], c["m"], _n(c)), g)
    else:
        d["B"] = _rhs(c, g)
        if c["kind"] == "grad":
            d["G"] = _gauss((c["s"], c["m"], _n(c)), g)
        elif c["kind"] == "rational":
            d["G"] = _gauss((c["m"], _n(c)), g)
    return d


def prepare(case, seed):
    st = _draw_inputs(case, seed)
    dims = (case["lx"], case["ly"], case["lz"], case["lt"])
    st["ctx"] = dsbcg.Context(dims, st["U"], case["kappa"])
    st["case"] = case
    if case["kind"] == "schur":
        st["ctx"].set_operator("schur")
    if case["kind"] in ("solve", "schur"):
        st["sigma"] = _shifts(case).numpy()
    elif case["kind"] in ("grad", "rational"):
        st["args"] = dict(dims=dims, kappa=case["kappa"], tol=case["tol"], storage=case["storage"], context=st["ctx"],
                          alpha0=ALPHA0, alpha=_weights(case).numpy())
        st["B"].requires_grad_(True)
        st["sigma"] = _shifts(case).requires_grad_(True)
        st["U"].requires_grad_(True)
    elif case["kind"] == "force":
        st["w"] = _weights(case).numpy()
    return st


def run(st):
    c, ctx = st["case"], st["ctx"]
    if c["kind"] == "apply":
        return ctx.apply(c["op"], st["B"], storage=c["storage"])
    if c["kind"] == "force":
        return ctx.force(st["X"], st["L"], st["w"], storage=c["storage"])
    if c["kind"] in ("solve", "schur"):
        return ctx.solve(st["B"], st["sigma"], c["tol"], storage=c["storage"])[0]
    if c["kind"] == "grad":
        out = dsbcg.DSBCGSolve.apply(st["B"], st["sigma"], st["U"], st["args"])
    else:
        ctx.update_gauge(st["U"].detach())
        out = dsbcg.DSBCGRational.apply(st["B"], st["sigma"], st["U"], st["args"])
    gB, gs, gU = torch.autograd.grad(out, (st["B"], st["sigma"], st["U"]), st["G"])
    return dict(out=out.detach(), gB=gB, gsigma=gs, gU=gU)


# ------------------------------------------------------------------ work --
def work(case):
    """Inputs once, outputs once (complex128 at the ABI; links once), and the operations: 1368 flop per site and field
    for one application of D (the usual count).  A solve's are those of the block process that these shifts and this
    tolerance take at least: about STEPS applications of A to m vectors, each with the m x m products per row of the
    basis (orthogonalisation) and of one shift's iterate."""
    c = case
    V, n, m, s = _volume(c), _n(c), c["m"], c["s"]
    links, block, d = 36 * 16.0 * V, 16.0 * m * n, 1368.0 * V * m
    if c["kind"] == "apply":
        return dict(bytes=2 * block + links, flops=d * (2 if c["op"] == "A" else 1))
    if c["kind"] == "force":
        # D on both blocks, then per link and field pair two spin projections and four outer products
        return dict(bytes=2 * s * block + 2 * links, flops=2 * d * s + 4 * V * m * s * 2 * (2 * 24 + 2 * 9 * 4 * 8.0))
    steps = 40.0 * (math.log10(1.0 / c["tol"]) / 8.0)
    one = steps * (2 * d + 8.0 * n * m * m * 4)
    if c["kind"] in ("solve", "schur"):
        return dict(bytes=block + links + s * block, flops=one)
    if c["kind"] == "grad":
        return dict(bytes=block + 2 * s * block + block + 2 * links, flops=(1 + s) * one + 2 * d * s)
    return dict(bytes=4 * block + 2 * links, flops=2 * one + 2 * d * s)


# ----------------------------------------------------------------- exact --
# Plain torch in 64 bits: the operator from its definition with half spinors, a shifted conjugate gradient, and the
# link gradient by torch's own differentiation of <lambda, A x>.
def _spin(k, l):
    """sigma_k on the spin index (-2) of a half spinor."""
    a, b = l[..., 0, :], l[..., 1, :]
    if k == 0:
        return torch.stack([b, a], dim=-2)
    if k == 1:
        return torch.stack([-1j * b, 1j * a], dim=-2)
    return torch.stack([a, -b], dim=-2)


def _colour(u, h):
    """(u h)[s, a] = sum_b u[a, b] h[s, b]"""
    return sum(u[..., None, :, b] * h[..., :, b, None] for b in range(3))


def _hop(psi, U):
    """sum_mu (1 - gamma_mu) U_mu(x) psi(x+mu) + (1 + gamma_mu) U_mu(x-mu)^H psi(x-mu); psi [m][t][z][y][x][4][3]."""
    out = None
    for mu in range(4):
        ax = -3 - mu                     # x, y, z, t axis of psi (and of U without its mu axis)
        u = U[..., mu, :, :]
        for sign in (-1, 1):             # forward hop: 1 - gamma; backward hop: 1 + gamma
            if sign < 0:
                p = torch.roll(psi, -1, dims=ax)
                if mu == 3:
                    p = torch.cat([p[:, :-1], -p[:, -1:]], dim=1)
            else:
                p = psi
            up, lo = p[..., 0:2, :], p[..., 2:4, :]
            if mu < 3:
                h = up + sign * 1j * _spin(mu, lo)
            else:
                h = up + sign * lo
            if sign < 0:
                h = _colour(u, h)
            else:
                h = torch.roll(_colour(u.mH, h), 1, dims=ax)
                if mu == 3:
                    h = torch.cat([-h[:, :1], h[:, 1:]], dim=1)
            low = -sign * 1j * _spin(mu, h) if mu < 3 else sign * h
            t = torch.cat([h, low], dim=-2)
            out = t if out is None else out + t
    return out


def _g5(psi):
    return torch.cat([-psi[..., 0:2, :], psi[..., 2:4, :]], dim=-2)


class _Exact:
    def __init__(self, c, U):
        self.c, self.U = c, U
        self.grid = (c["lt"], c["lz"], c["ly"], c["lx"], 4, 3)
        if c["kind"] == "schur":
            ar = [torch.arange(L, device="cuda") for L in self.grid[:4]]
            par = (ar[0][:, None, None, None] + ar[1][:, None, None] + ar[2][:, None] + ar[3]) & 1
            self.odd = torch.nonzero(par.reshape(-1) == 1).reshape(-1)

    def field(self, v):
        if self.c["kind"] != "schur":
            return v.reshape((v.shape[0],) + self.grid)
        f = torch.zeros((v.shape[0], _volume(self.c), 12), dtype=v.dtype, device=v.device)
        f[:, self.odd] = v.reshape(v.shape[0], -1, 12)
        return f.reshape((v.shape[0],) + self.grid)

    def vector(self, f):
        f = f.reshape(f.shape[0], -1, 12)
        return (f if self.c["kind"] != "schur" else f[:, self.odd]).reshape(f.shape[0], -1)

    def Df(self, psi):
        k = self.c["kappa"]
        if self.c["kind"] == "schur":
            return psi - k * k * _hop(_hop(psi, self.U), self.U)
        return psi - k * _hop(psi, self.U)

    def op(self, name, v):
        psi = self.field(v)
        if name != "Ddag":
            psi = self.Df(psi)
        if name != "D":
            psi = _g5(self.Df(_g5(psi)))
        return self.vector(psi)

    def solve(self, B, sigma):
        """Conjugate gradients for every shift on one Krylov space per right-hand side (base: the smallest shift);
        each shifted system stops when its residual is below 1e-15 of the right-hand side."""
        s0, s = float(sigma.min()), sigma.numel()
        delta = (sigma - s0).to(B.device)
        dot = lambda a, b: (torch.view_as_real(a) * torch.view_as_real(b)).sum((-1, -2))
        r, p, bb = B.clone(), B.clone(), dot(B, B)
        rr = bb.clone()
        X = torch.zeros((s,) + tuple(B.shape), dtype=B.dtype, device=B.device)
        P = B.expand(X.shape).clone()
        one = torch.ones_like(rr)
        alpha_old, beta_old = one.clone(), torch.zeros_like(rr)
        z, z_old = torch.ones((s, B.shape[0]), dtype=torch.float64, device=B.device), None
        z_old = z.clone()
        on = list(range(s))
        for it in range(1500):
            q = self.op("A", p) + s0 * p
            alpha = rr / dot(p, q)
            d = delta[:, None]
            z_new = z * z_old * alpha_old / (alpha * beta_old * (z_old - z) + z_old * alpha_old * (1 + alpha * d))
            x_step = alpha * z_new / z
            for j in on:
                X[j] += x_step[j, :, None] * P[j]
            r = r - alpha[:, None] * q
            rn = dot(r, r)
            beta = rn / rr
            for j in on:
                P[j] *= (beta * (z_new[j] / z[j]) ** 2)[:, None]
                P[j] += z_new[j, :, None] * r
            p = r + beta[:, None] * p
            z_old, z, alpha_old, beta_old, rr = z, z_new, alpha, beta, rn
            if it % 8 == 7:
                rel = (z.abs() * (rr / bb).sqrt()).max(dim=1).values.tolist()
                for j in [j for j in on if not rel[j] > 1e-15]:
                    on.remove(j)
                    z[j], z_old[j] = 1.0, 1.0        # out of use: kept away from underflow
                    delta[j] = 0.0
                if not on:
                    break
        return X

    def link_gradient(self, pairs):
        """-d/dU Re <lambda, A(U) x> summed over (lambda, x, weight) blocks, in the dRe + i dIm convention."""
        U, total = self.U, torch.zeros_like(self.U)
        for lam, x, w in pairs:
            self.U = U.detach().clone().requires_grad_(True)
            a, b = self.Df(self.field(lam)), self.Df(self.field(x))
            loss = -w * (torch.view_as_real(a) * torch.view_as_real(b)).sum()
            total += torch.autograd.grad(loss, self.U)[0]
        self.U = U
        return total


def exact(case, seed):
    c = case
    V = _volume(c)
    if c["kind"] not in ("apply", "force") and V * c["m"] * (c["s"] + 8) > 45e6:
        return None                       # a solve on the largest lattices takes too long here
    d = _draw_inputs(c, seed)
    e = _Exact(c, d["U"])
    if c["kind"] == "apply":
        out = torch.empty_like(d["B"])
        for i in range(0, c["m"], 4):
            out[i:i + 4] = e.op(c["op"], d["B"][i:i + 4])
        return out
    if c["kind"] == "force":
        w = _weights(c).tolist()
        return e.link_gradient((d["L"][j, i:i + 4], d["X"][j, i:i + 4], w[j])
                               for j in range(c["s"]) for i in range(0, c["m"], 4))
    sigma = _shifts(c)
    X = e.solve(d["B"], sigma)
    if c["kind"] in ("solve", "schur"):
        return X
    if c["kind"] == "grad":
        L = torch.stack([e.solve(d["G"][j], sigma[j:j + 1])[0] for j in range(c["s"])])
        out, gB = X, L.sum(0)
    else:
        a = _weights(c).to(X.device)[:, None, None]
        L = a * e.solve(d["G"], sigma)
        out, gB = ALPHA0 * d["B"] + (a * X).sum(0), ALPHA0 * d["G"] + L.sum(0)
    gs = -(torch.view_as_real(L) * torch.view_as_real(X)).sum((-1, -2, -3)).cpu()
    gU = e.link_gradient((L[j], X[j], 1.0) for j in range(c["s"]))
    return dict(out=out, gB=gB, gsigma=gs, gU=gU)

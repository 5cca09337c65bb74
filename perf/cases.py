"""The calls that a user of this framework makes, as measurable cases.

Every case goes through the public entry points (``binding``, ``autograd``): the operator H(mu)
alone, sgn(H) b by the two-sided Lanczos method, its gauge-force VJP, Theorem 1's directional
derivative, the nested form and the uneven batch.  Lattices, sources, Krylov sizes, projection
schedules and link roughness are those of the benchmark's workloads and of the tests.  The Wilson
mass is -1 (the well-conditioned point of the tests and of the benchmark's mixed leg): at -2 the
k-step map amplifies one rounding error to 1e-4 and more in dU, so that no two correct programs
agree there; the work per step does not depend on the mass.
"""
from __future__ import annotations

import math

import torch

from paper_1604_08057_gb300 import autograd, binding

_C = torch.complex128
M_W = -1.0


def _case(name, kind, dims, nsrc, k=0, precision="fp64", rebiorth=1, passes=2, mu=0.3, eps=0.2, **more):
    nx, ny, nz, nt = dims
    return dict(name=name, kind=kind, nx=nx, ny=ny, nz=nz, nt=nt, nsrc=nsrc, k=k, precision=precision,
                rebiorth=rebiorth, passes=passes, mu=mu, eps=eps, **more)


def listed():
    return [
        # one operator application on the smallest workload lattice: latency and launches
        _case("apply_h 4x4^3", "apply", (4, 4, 4, 4), 1, eps=0.3, dagger=False),
        # the multi-source FP32 operator of the benchmark's D_w leg (32 sources share the links)
        _case("apply_h 14x14^3 x32 mixed", "apply", (14, 14, 14, 14), 32, precision="mixed", dagger=False),
        # the FP64 adjoint operator on the 16-source workload's lattice
        _case("apply_h_dag 6x18^3 x16", "apply", (18, 18, 18, 6), 16, mu=0.5, dagger=True),
        # sgn(H) b on the four-source workload (projections every 20 steps, one pass)
        _case("sign 8x8^3 x4 k400", "sign", (8, 8, 8, 8), 4, 400, rebiorth=20, passes=1, mu=0.2, eps=0.25),
        # sgn(H) b at the largest lattice with the paper's nested k x k stage (inner size 100)
        _case("sign nested 14x14^3 k800", "nested", (14, 14, 14, 14), 1, 800, rebiorth=60, passes=1, inner=100),
        # sgn(H) b with FP32 vectors, several sources, the library's default schedule (every step, two passes)
        _case("sign mixed 6x18^3 x4 k80", "sign", (18, 18, 18, 6), 4, 80, precision="mixed", mu=0.5),
        # forward and gauge force on the smallest workload: the latency-bound end of the headline call
        _case("vjp 4x4^3 k200", "vjp", (4, 4, 4, 4), 1, 200, rebiorth=20, passes=1, eps=0.3),
        # the headline call: sgn(H) b with its gauge force at the largest lattice
        _case("vjp 14x14^3 k800", "vjp", (14, 14, 14, 14), 1, 800, rebiorth=60, passes=1),
        # the same through torch.autograd with default options, on the batch's middle lattice
        _case("autograd 6x12^3 k120", "autograd", (12, 12, 12, 6), 1, 120, mu=0.1),
        # Theorem 1: one directional derivative along links and mu, on a lattice with odd sides
        _case("jvp 9x7x5x11 x2 k150", "jvp", (11, 5, 7, 9), 2, 150, rebiorth=20, passes=1, eps=0.25),
        # the uneven batch: forward and force of eight problems on three lattices, four workers
        _case("batch of 8", "batch", (8, 8, 8, 8), 1, 160, rebiorth=20, passes=1, problems=8),
    ]


def _unnamed(case):
    del case["name"]
    return case


_KINDS = ("apply", "apply", "sign", "nested", "vjp", "vjp", "autograd", "jvp", "batch")


def draw(rng):
    kind = rng.choice(_KINDS)
    precision = "mixed" if kind in ("apply", "sign") and rng.random() < 0.35 else "fp64"
    # the derivative kinds stay where the unconverged k-step map is well conditioned
    mu = rng.choice((0.1, 0.2) if kind in ("vjp", "autograd", "jvp", "batch") else (0.1, 0.2, 0.3, 0.5))
    eps = 0.2 if kind in ("vjp", "autograd", "jvp", "batch") else rng.choice((0.2, 0.25, 0.3))

    def log(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    while True:
        side = math.exp(rng.uniform(math.log(4.0), math.log(15.0)))
        dims = tuple(max(3, min(18, int(round(side * rng.uniform(0.75, 1.3))))) for _ in range(4))
        v = math.prod(dims)
        if not 128 <= v <= 40000:
            continue
        if kind == "apply":
            nsrc = rng.choice((1, 2, 3, 4, 7, 16, 32))
            return _unnamed(_case("", kind, dims, nsrc, precision=precision, mu=mu, eps=eps,
                                  dagger=rng.random() < 0.5))
        nsrc = rng.choice((1, 1, 2, 3, 4)) if kind in ("sign", "vjp", "jvp") else 1
        reb, passes = rng.choice(((1, 2), (20, 1), (20, 1), (10, 1)))
        k = log(20, 80) if precision == "mixed" else log(30, min(v // 2, 400))
        more = {}
        if kind == "nested":
            more["inner"] = min(k, log(30, 120))
        if kind == "batch":
            more["problems"] = rng.randint(2, 6)
            if v > 8 ** 4:
                continue
        case = _unnamed(_case("", kind, dims, nsrc, k, precision, reb, passes, mu, eps, **more))
        if work(case)["flops"] < 5e11:
            return case


# ---- inputs -----------------------------------------------------------------------------------

def _links(dims, eps, gen):
    """U = expm(i eps A), A a Gaussian traceless Hermitian matrix, shape (Nt, Nz, Ny, Nx, 4, 3, 3)."""
    nx, ny, nz, nt = dims
    xi = torch.randn((nt, nz, ny, nx, 4, 8), generator=gen, device="cuda", dtype=torch.float64) * 0.5
    a = torch.zeros(xi.shape[:-1] + (3, 3), device="cuda", dtype=_C)
    for n, (i, j) in enumerate(((0, 1), (0, 2), (1, 2))):
        a[..., i, j] = torch.complex(xi[..., 2 * n], -xi[..., 2 * n + 1])
        a[..., j, i] = torch.complex(xi[..., 2 * n], xi[..., 2 * n + 1])
    d, e = xi[..., 6], xi[..., 7] / math.sqrt(3.0)
    a[..., 0, 0] = d + e
    a[..., 1, 1] = e - d
    a[..., 2, 2] = -2.0 * e
    return torch.linalg.matrix_exp(1j * eps * a).contiguous()


def _spinors(dims, nsrc, gen):
    nx, ny, nz, nt = dims
    z = torch.randn((nsrc, nt, nz, ny, nx, 4, 3, 2), generator=gen, device="cuda", dtype=torch.float64)
    return torch.view_as_complex(z / math.sqrt(2.0))


def _problems(case):
    """(dims, mu, k) of the batch's problems: three lattices, three mu, k between 0.4 and 1 of the largest."""
    dims = (case["nx"], case["ny"], case["nz"], case["nt"])
    half = tuple(max(3, d // 2) for d in dims)
    mid = tuple(max(3, (3 * d) // 4) for d in dims)
    out = []
    for i in range(case["problems"]):
        d = (dims, mid, half)[i % 3]
        k = int(case["k"] * (0.4 + 0.6 * ((7 * i) % 8) / 7.0))
        out.append((d, (0.1, 0.3, 0.5)[(i // 3) % 3], max(20, min(k, math.prod(d) // 2))))
    return out


def prepare(case, seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    s = dict(case)
    dims = (case["nx"], case["ny"], case["nz"], case["nt"])
    if case["kind"] == "batch":
        s["list"] = [dict(u=_links(d, case["eps"], gen), mu=mu, m_w=M_W, b=_spinors(d, 1, gen)[0], k=k,
                          xbar=_spinors(d, 1, gen)[0]) for d, mu, k in _problems(case)]
        return s
    s["u"] = _links(dims, case["eps"], gen)
    s["b"] = _spinors(dims, case["nsrc"], gen)
    if case["kind"] in ("vjp", "autograd"):
        s["xbar"] = _spinors(dims, case["nsrc"], gen)
    if case["kind"] == "jvp":
        s["e"] = torch.view_as_complex(torch.randn(tuple(s["u"].shape) + (2,), generator=gen, device="cuda",
                                                   dtype=torch.float64))
    return s


def run(s):
    kind = s["kind"]
    opt = dict(precision=s["precision"], rebiorth=s["rebiorth"], passes=s["passes"])
    if kind == "apply":
        return binding.apply_H(s["u"], s["mu"], M_W, s["b"], dagger=s["dagger"], precision=s["precision"])
    if kind == "sign":
        return binding.tsl_sign(s["u"], s["mu"], M_W, s["b"], s["k"], **opt)
    if kind == "nested":
        binding.nested_sign(s["inner"], **opt)
        try:
            return binding.tsl_sign(s["u"], s["mu"], M_W, s["b"], s["k"], **opt)
        finally:
            binding.nested_sign(0, **opt)
    if kind == "vjp":
        du, dmu, x = binding.tsl_sign_vjp(s["u"], s["mu"], M_W, s["b"], s["k"], s["xbar"], **opt)
        return du, dmu, x
    if kind == "autograd":
        u = s["u"].detach().requires_grad_(True)
        mu = torch.tensor(s["mu"], dtype=torch.float64, device="cuda", requires_grad=True)
        x = autograd.tsl_sign(u, mu, s["b"], s["k"], M_W, **opt)
        x.backward(s["xbar"])
        return u.grad, mu.grad.item(), x.detach()
    if kind == "jvp":
        return binding.tsl_sign_jvp(s["u"], s["mu"], M_W, s["b"], s["k"], e=s["e"], m_dir=0.7, **opt)
    res = binding.tsl_batch(s["list"], nworkers=4, **opt)
    return [(r["dU"], r["dmu"], r["x"]) for r in res]


# ---- what a pass cannot do without ------------------------------------------------------------

_H = 1368.0                                   # flops of H or H^dagger per site


def _projections(k, period):
    """Basis vectors (V and W together) that the Gram-Schmidt steps of one forward pass read."""
    steps = [j for j in range(1, k) if period == 1 or (period > 1 and j % period < 2)]
    return 2.0 * sum(steps)


def _tsl_work(v, nsrc, k, rebiorth, passes, vjp, block):
    half = 2.0 if block else 1.0
    per_step = (2 * half + (1 if block else 0) * 2) * _H + 11 * 96 * half     # H, H^dagger (and dH), update, scales
    proj = _projections(k, rebiorth) * passes * 2 * 96 * half                 # dots and updates
    flops = v * (k * per_step + proj + 96.0 * k * half) + 8.0 * k ** 3
    if vjp:
        # the adjoint recurrence (two H, its combinations), two force terms per step, the adjoint projections
        flops += v * (k * (2 * _H + 18 * 96 + 2 * 8 * 9 * 16) + _projections(k, rebiorth) * 3 * 96) + 16.0 * k ** 3
    return nsrc * flops


def work(case):
    kind, nsrc, k = case["kind"], case["nsrc"], case["k"]
    if kind == "batch":
        b = f = 0.0
        for d, _, kk in _problems(case):
            v = math.prod(d)
            b += v * (2 * 576 + 3 * 192)
            f += _tsl_work(v, 1, kk, case["rebiorth"], case["passes"], True, False)
        return {"bytes": b, "flops": f}
    v = case["nx"] * case["ny"] * case["nz"] * case["nt"]
    byt = v * (576.0 + 2 * 192.0 * nsrc)                    # links, b, x
    if kind == "apply":
        return {"bytes": byt, "flops": v * nsrc * _H}
    if kind in ("vjp", "autograd"):
        byt += v * (576.0 + 192.0 * nsrc)                   # dU, xbar
    if kind == "jvp":
        byt += v * (576.0 + 192.0 * nsrc)                   # E, dx
    return {"bytes": byt, "flops": _tsl_work(v, nsrc, k, case["rebiorth"], case["passes"],
                                             kind in ("vjp", "autograd"), kind == "jvp")}


# ---- the same in 64 bits, in plain torch ------------------------------------------------------

def _hop(psi, m, nu, sign):
    """(1 + sign gamma_nu) m psi with psi already shifted; psi (n, Nt, Nz, Ny, Nx, 4, 3)."""
    p0, p1, p2, p3 = psi.unbind(-2)
    if nu == 0:
        h0, h1 = p0 - sign * 1j * p3, p1 - sign * 1j * p2
    elif nu == 1:
        h0, h1 = p0 - sign * p3, p1 + sign * p2
    elif nu == 2:
        h0, h1 = p0 - sign * 1j * p2, p1 + sign * 1j * p3
    else:
        h0, h1 = p0 + sign * p2, p1 + sign * p3
    g = (m.unsqueeze(-3) * torch.stack((h0, h1), -2).unsqueeze(-2)).sum(-1)      # m_ab h_sb
    g0, g1 = g.unbind(-2)
    if nu == 0:
        l0, l1 = sign * 1j * g1, sign * 1j * g0
    elif nu == 1:
        l0, l1 = sign * g1, -sign * g0
    elif nu == 2:
        l0, l1 = sign * 1j * g0, -sign * 1j * g1
    else:
        l0, l1 = sign * g0, sign * g1
    return torch.stack((g0, g1, l0, l1), -2)


class _Op:
    """H(mu) = gamma5 D_w(mu) and its adjoint gamma5 D_w(-mu) for fixed links."""

    def __init__(self, u, mu):
        self.f = [u[..., nu, :, :] for nu in range(4)]
        self.b = [torch.roll(u[..., nu, :, :], 1, 3 - nu).mH for nu in range(4)]
        self.mu = mu
        self.kappa = 1.0 / (2.0 * M_W + 8.0)

    def hops(self, psi, mu, fwd=None, bwd=None):
        acc = 0.0
        for nu in range(4):
            up, dn = (torch.exp(mu), torch.exp(-mu)) if nu == 3 else (1.0, 1.0)
            ax = 4 - nu
            acc = acc + up * _hop(torch.roll(psi, -1, ax), (fwd or self.f)[nu], nu, 1.0)
            acc = acc + dn * _hop(torch.roll(psi, 1, ax), (bwd or self.b)[nu], nu, -1.0)
        return acc

    def __call__(self, psi, dagger=False):
        y = psi - self.kappa * self.hops(psi, -self.mu if dagger else self.mu)
        return torch.cat((y[..., :2, :], -y[..., 2:, :]), -2)


def _sgn(t):
    """Newton iteration for the matrix sign with Frobenius-norm scaling while it helps."""
    x = t
    for it in range(60):
        xi = torch.linalg.inv(x)
        g = 1.0
        if it < 8:
            g = ((torch.linalg.norm(xi) / torch.linalg.norm(x)).detach()) ** 0.5
        new = 0.5 * (g * x + xi / g)
        step = float(torch.linalg.norm(new.detach() - x.detach()) / torch.linalg.norm(new.detach()))
        x = new
        if it > 8 and step < 1e-13:
            break
    return x


def _lanczos(mv, mvd, r, s, beta0, sw, k, period, passes):
    """x = beta0 V_k sgn(T_k) e_1 by k steps of two-sided Lanczos from r/beta0 and sw s (flat fields)."""
    vs, ws, al, be, de = [], [], [], [], []
    v, w = r / beta0, s * sw
    bt = dl = None
    for j in range(k):
        vs.append(v)
        ws.append(w)
        p = mv(v)
        a = torch.sum(w.conj() * p)
        al.append(a)
        if j == k - 1:
            break
        r = p - a * v
        s = mvd(w) - a.conj() * w
        if j > 0:
            r = r - bt * vs[-2]
            s = s - dl * ws[-2]
        if period == 1 or (period > 1 and (j + 1) % period < 2):
            for _ in range(passes):
                vm, wm = torch.stack(vs), torch.stack(ws)
                c, d = wm.conj() @ r, vm.conj() @ s
                r, s = r - c @ vm, s - d @ wm
        om = torch.sum(s.conj() * r)
        dl = torch.sqrt(torch.abs(om))
        bt = om / dl
        be.append(bt)
        de.append(dl.to(_C))
        v, w = r / dl, s / bt.conj()
    t = torch.diag(torch.stack(al)) + torch.diag(torch.stack(be), 1) + torch.diag(torch.stack(de), -1)
    y = beta0 * _sgn(t)[:, 0]
    return y @ torch.stack(vs)


def _sign_one(u, mu, b, k, period, passes):
    op = _Op(u, mu)
    shape = (1,) + tuple(b.shape)
    mv = lambda p: op(p.reshape(shape)).reshape(-1)                  # noqa: E731
    mvd = lambda p: op(p.reshape(shape), True).reshape(-1)           # noqa: E731
    f = b.reshape(-1)
    n = torch.linalg.norm(f)
    return _lanczos(mv, mvd, f, f, n, 1.0 / n, k, period, passes).reshape(b.shape)


def _grad_one(u, mu, b, xbar, k, period, passes):
    u = u.detach().requires_grad_(True)
    m = torch.tensor(mu, dtype=torch.float64, device="cuda", requires_grad=True)
    x = _sign_one(u, m, b, k, period, passes)
    gu, gm = torch.autograd.grad(x, (u, m), xbar)
    return gu, float(gm), x.detach()


def _jvp_one(u, mu, b, e, md, k, period, passes):
    op, shape, n = _Op(u, mu), (1,) + tuple(b.shape), b.numel()
    ef = [e[..., nu, :, :] for nu in range(4)]
    eb = [torch.roll(e[..., nu, :, :], 1, 3 - nu).mH for nu in range(4)]

    def dh(p, dagger):
        m = -mu if dagger else mu
        acc = op.hops(p, m, ef, eb)
        md_ = -md if dagger else md
        acc = acc + md_ * torch.exp(m) * _hop(torch.roll(p, -1, 1), op.f[3], 3, 1.0)
        acc = acc - md_ * torch.exp(-m) * _hop(torch.roll(p, 1, 1), op.b[3], 3, -1.0)
        y = -op.kappa * acc
        return torch.cat((y[..., :2, :], -y[..., 2:, :]), -2)

    def mv(z):
        t, l = z[:n].reshape(shape), z[n:].reshape(shape)
        return torch.cat(((op(t) + dh(l, False)).reshape(-1), op(l).reshape(-1)))

    def mvd(z):
        t, l = z[:n].reshape(shape), z[n:].reshape(shape)
        return torch.cat((op(t, True).reshape(-1), (dh(t, True) + op(l, True)).reshape(-1)))

    f = b.reshape(-1)
    r, s = torch.cat((torch.zeros_like(f), f)), torch.cat((f, f))
    beta0 = torch.linalg.norm(r)
    sw = beta0 / torch.sum(s.conj() * r).conj()
    z = _lanczos(mv, mvd, r, s, beta0, sw, k, period, passes)
    return z[:n].reshape(b.shape), z[n:].reshape(b.shape)


def _too_long(case):
    """Whether exact() would take over about 20 seconds, or (reverse mode) over about 100 GB of saved tensors."""
    v, k, nsrc = case["nx"] * case["ny"] * case["nz"] * case["nt"], case["k"], case["nsrc"]
    grad = case["kind"] in ("vjp", "autograd", "batch")
    if grad and v * 192.0 * (_projections(k, case["rebiorth"]) * case["passes"] + 80.0 * k) > 1e11:
        return True
    if case["kind"] == "batch":
        return sum(6.0 * kk * (3e-3 + 1e-7 * math.prod(d)) for d, _, kk in _problems(case)) > 20.0
    return (6.0 if grad else 2.0) * k * nsrc * (3e-3 + 1e-7 * v) > 20.0


def exact(case, seed):
    if _too_long(case):
        return None
    s = prepare(case, seed)
    kind, k, per, ps = case["kind"], case["k"], case["rebiorth"], case["passes"]
    mu = torch.tensor(case["mu"], dtype=torch.float64, device="cuda")
    if kind == "apply":
        op = _Op(s["u"], mu)
        return torch.cat([op(b[None], case["dagger"]) for b in s["b"]])
    if kind in ("sign", "nested"):
        return torch.stack([_sign_one(s["u"], mu, b, k, per, ps) for b in s["b"]])
    if kind in ("vjp", "autograd"):
        one = [_grad_one(s["u"], case["mu"], b, xb, k, per, ps) for b, xb in zip(s["b"], s["xbar"])]
        return sum(o[0] for o in one), sum(o[1] for o in one), torch.stack([o[2] for o in one])
    if kind == "jvp":
        one = [_jvp_one(s["u"], mu, b, s["e"], 0.7, k, per, ps) for b in s["b"]]
        return torch.stack([o[0] for o in one]), torch.stack([o[1] for o in one])
    return [_grad_one(p["u"], p["mu"], p["b"], p["xbar"], p["k"], per, ps) for p in s["list"]]

"""The workloads this library is timed on: what its users have it do, through its public entry points.

A case is one call (or one step of several calls) of a user's program on seeded synthetic lattices: links
U = exp(iA) with A traceless Hermitian Gaussian (sigma 0.25 or 0.3, as in the library's presets), complex-Gaussian
sources, kappa 0.12 to 0.156, antiperiodic in time.  Solves run to a relative true residual of 1e-11 (1e-12 inside
a trajectory), a decade or two below the 1e-10 the library's tests use, so that a solution is determined to about
1e-10 whatever the rounding on the way there.
"""
import math

import torch

import paper_1207_2223_gb300 as lq
from paper_1207_2223_gb300.autograd import pseudofermion_action

DEV = "cuda"
TOL = 1e-11


# ------------------------------------------------------------------ the cases

def _case(name, kind, dims, **more):
    c = {"name": name, "kind": kind, "lx": dims[0], "ly": dims[1], "lz": dims[2], "lt": dims[3],
         "kappa": 0.15, "sigma": 0.3}
    c.update(more)
    return c


def listed():
    return [
        # smallest call: M^dag M on the caller's buffers without a context (a program that owns all device memory)
        _case("static_mdagm_8x8x8x8", "static", (8, 8, 8, 8)),
        # one FP64 application of M^dag on an odd-sized lattice (residual checks, phi = M^dag chi of a heat bath)
        _case("apply_m_f64_15x16x17x18", "apply_m", (15, 16, 17, 18), dagger=True),
        # FP64 M^dag M on the large lattice: checking a solution that came from elsewhere
        _case("apply_mdagm_f64_32x32x32x64", "apply_mdagm", (32, 32, 32, 64), kappa=0.156, sigma=0.25),
        # plain FP64 CG, the default precision of the solver
        _case("solve_f64_16x16x16x16", "solve", (16, 16, 16, 16), kappa=0.155, prec="f64", load=False),
        # the large measurement: load a configuration, solve for one source with FP16 storage
        _case("solve_f16_32x32x32x64", "solve", (32, 32, 32, 64), kappa=0.156, sigma=0.25, prec="f16_12", load=True),
        # mixed solve with FP32 storage on a ragged lattice, links already loaded
        _case("solve_f32_12_14x18x20x26", "solve", (14, 18, 20, 26), kappa=0.152, prec="f32_12", load=False),
        # mixed solve of the size a small molecular-dynamics run makes thousands of
        _case("solve_f16_8x8x8x8", "solve", (8, 8, 8, 8), prec="f16_12", load=False),
        # propagator: 12 spin-colour sources on one gauge field
        _case("batch_f16_20x20x20x20_12rhs", "batch", (20, 20, 20, 20), kappa=0.154, prec="f16_12", nrhs=12),
        # independent lattices of uneven size and kappa solved together (8^4, 12^4, 16^4, 8^3 x 16)
        _case("batch_f32_12_uneven", "uneven", (8, 8, 8, 16), kappa=0.155, prec="f32_12", mid=12, large=16),
        # a whole trajectory: heat bath, leapfrog, Metropolis, with mixed solves
        _case("hmc_f16_8x8x8x8", "hmc", (8, 8, 8, 8), prec="f16_12", steps=10, beta=5.6),
        # differentiable pseudofermion action, forward and backward, at its default FP64 precision
        _case("autograd_f64_12x12x12x12", "autograd", (12, 12, 12, 12)),
        # molecular dynamics outside the solve: both forces, the link update, links in and out
        _case("md_24x24x24x32", "md", (24, 24, 24, 32), beta=5.6),
    ]


def _extents(rng, lo, hi):
    """Four extents whose product is spread over [lo, hi] on a logarithmic scale, odd ones among them."""
    target = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    side = target ** 0.25
    d = [max(3, round(side * math.exp(rng.uniform(-0.25, 0.25)))) for _ in range(3)]
    d.append(max(3, round(target / (d[0] * d[1] * d[2]))))
    return tuple(d)


def draw(rng):
    kind = rng.choice(["static", "apply_m", "apply_mdagm", "solve", "solve", "solve", "batch", "uneven", "hmc",
                       "autograd", "md"])
    kappa, sigma = round(rng.uniform(0.12, 0.152), 4), round(rng.uniform(0.25, 0.3), 3)
    mixed = ["f32", "f32_12", "f16_12", "bf16_12", "i16_12"]
    c = {"kind": kind}
    if kind == "static":
        dims = _extents(rng, 256, 50000)
    elif kind in ("apply_m", "apply_mdagm"):
        dims = _extents(rng, 256, 1500000)
        if kind == "apply_m":
            c["dagger"] = rng.random() < 0.5
    elif kind == "solve":
        c["prec"] = rng.choice(["f64"] + mixed)
        dims = _extents(rng, 256, 60000 if c["prec"] == "f64" else 800000)
        c["load"] = rng.random() < 0.5
    elif kind == "batch":
        c["prec"], c["nrhs"] = rng.choice(mixed), rng.choice([2, 3, 4, 6, 12])
        dims = _extents(rng, 256, 400000 // c["nrhs"])
    elif kind == "uneven":
        c["prec"], c["mid"], c["large"] = rng.choice(mixed), rng.randint(5, 12), rng.randint(6, 16)
        dims = _extents(rng, 256, 8000)
    elif kind == "hmc":
        c["prec"], c["steps"], c["beta"] = rng.choice(["f64", "f32_12", "f16_12"]), rng.randint(6, 16), 5.6
        dims = _extents(rng, 256, 4000)
    elif kind == "autograd":
        dims = _extents(rng, 256, 20000)
    else:
        dims, c["beta"] = _extents(rng, 256, 400000), 5.6
    return dict(c, lx=dims[0], ly=dims[1], lz=dims[2], lt=dims[3], kappa=kappa, sigma=sigma)


def _dims(c):
    return (c["lx"], c["ly"], c["lz"], c["lt"])


def _systems(c):
    """(dims, kappa) of every lattice of the case."""
    if c["kind"] != "uneven":
        return [(_dims(c), c["kappa"])]
    m, n, h = c["mid"], c["large"], min(c["lx"], c["ly"], c["lz"])
    return [((h, h, h, h), 0.12), ((m, m, m, m), 0.14), ((n, n, n, n), 0.15), (_dims(c), c["kappa"])]


# ------------------------------------------------------------------ inputs

def _gauge(dims, sigma, gen, chunk=1 << 20):
    """exp(iA) with N(0, sigma^2) entries of a traceless Hermitian A, complex128 [V][4][3][3]."""
    n = 4 * math.prod(dims)
    U = torch.empty((n, 3, 3), dtype=torch.complex128, device=DEV)
    for lo in range(0, n, chunk):
        k = min(chunk, n - lo)
        g = sigma * torch.randn((k, 9), dtype=torch.float64, device=DEV, generator=gen)
        A = torch.zeros((k, 3, 3), dtype=torch.complex128, device=DEV)
        for i in range(3):
            A[:, i, i] = g[:, i] - g[:, :3].mean(1)
        for (i, j), m in (((0, 1), 3), ((0, 2), 5), ((1, 2), 7)):
            A[:, i, j] = torch.complex(g[:, m], g[:, m + 1])
            A[:, j, i] = torch.complex(g[:, m], -g[:, m + 1])
        U[lo:lo + k] = torch.matrix_exp(1j * A)
    # rows orthonormalised, the third rebuilt, so that the 12-real formats hold the same links
    r0 = U[:, 0] / torch.linalg.vector_norm(U[:, 0], dim=1, keepdim=True)
    r1 = U[:, 1] - (r0.conj() * U[:, 1]).sum(1, keepdim=True) * r0
    r1 = r1 / torch.linalg.vector_norm(r1, dim=1, keepdim=True)
    U[:, 0], U[:, 1], U[:, 2] = r0, r1, torch.linalg.cross(r0, r1).conj()
    return U.view(-1, 4, 3, 3)


def _spinor(dims, gen, n=None):
    shape = ((n,) if n else ()) + (math.prod(dims), 4, 3, 2)
    return torch.view_as_complex(torch.randn(shape, dtype=torch.float64, device=DEV, generator=gen) * 0.5 ** 0.5)


class _State:
    """What a user's program keeps: contexts with their links, sources and result buffers."""

    def __init__(self, case):
        self.case, self.ctxs = case, []

    def context(self, dims, U):
        ctx = lq.lq_create(dims)
        self.ctxs.append(ctx)
        if U is not None:
            lq.lq_gauge_set(ctx, U)
        return ctx

    def __del__(self):
        for ctx in self.ctxs:
            lq.lq_destroy(ctx)


def prepare(case, seed):
    gen = torch.Generator(device=DEV)
    gen.manual_seed(1000003 * seed + 17)
    s, kind = _State(case), case["kind"]
    s.seed = seed % (1 << 30)
    systems = _systems(case)
    s.U = [_gauge(d, case["sigma"], gen) for d, _ in systems]
    s.phi = [_spinor(d, gen, case.get("nrhs")) for d, _ in systems]
    s.x = [torch.zeros_like(p) for p in s.phi]
    dims = systems[0][0]
    if kind in ("static", "autograd"):
        pass
    elif kind in ("hmc", "md"):
        s.context(dims, None)
        s.p = torch.randn((math.prod(dims), 4, 8), dtype=torch.float64, device=DEV, generator=gen)
        s.F, s.Ff, s.Uout = torch.empty_like(s.p), torch.empty_like(s.p), torch.empty_like(s.U[0])
    else:
        for (d, _), U in zip(systems, s.U):
            s.context(d, U)
    return s


# ------------------------------------------------------------------ one pass

def run(s):
    c = s.case
    kind, kappa, dims = c["kind"], c["kappa"], _dims(c)
    prec = lq.PRECISIONS[c.get("prec", "f64")]
    U, phi, x = s.U[0], s.phi[0], s.x[0]
    if kind == "static":
        lq.lq_apply_MdagM_static(x, U, phi, dims, kappa)
        return x
    if kind == "autograd":
        Ua, pa = U.detach().requires_grad_(True), phi.detach().requires_grad_(True)
        S = pseudofermion_action(Ua, pa, dims, kappa, TOL)
        S.backward()
        return {"S": S.detach(), "dU": Ua.grad, "dphi": pa.grad}
    ctx = s.ctxs[0]
    if kind == "apply_m":
        lq.lq_apply_M(ctx, x, phi, kappa, c["dagger"], prec)
        return x
    if kind == "apply_mdagm":
        lq.lq_apply_MdagM(ctx, x, phi, kappa, prec)
        return x
    if kind == "solve":
        if c["load"]:
            lq.lq_gauge_set(ctx, U)
        lq.lq_solve_MdagM(ctx, x, phi, kappa, TOL, 20000, prec, 50)
        return x
    if kind in ("batch", "uneven"):
        lq.lq_solve_batch(s.ctxs, s.x, s.phi, [k for _, k in _systems(c)], c.get("nrhs", 1), TOL, 20000, prec, 50)
        return list(s.x)
    if kind == "hmc":
        lq.lq_gauge_set(ctx, U)
        r = lq.lq_hmc_trajectory_seeded(ctx, s.seed, 0, c["beta"], kappa, c["steps"], 1.0, 1e-12, 20000, prec, 50,
                                        p_out=s.p)
        lq.lq_gauge_get(ctx, s.Uout)
        return {"U": s.Uout, "p": s.p, "accepted": r["accepted"], "plaquette": r["plaquette"],
                "dH": torch.tensor([r["dH"], r["dK"], r["dSg"], r["dSf"]], dtype=torch.float64)}
    # molecular dynamics step outside the solve: phi stands for the solution X
    lq.lq_gauge_set(ctx, U)
    action = lq.lq_gauge_action(ctx, c["beta"])
    lq.lq_gauge_force(ctx, s.F, c["beta"])
    lq.lq_fermion_force(ctx, s.Ff, phi, kappa)
    lq.lq_link_update(ctx, s.p, 0.05)
    lq.lq_gauge_get(ctx, s.Uout)
    return {"F": s.F, "Ff": s.Ff, "U": s.Uout, "action": action}


# ------------------------------------------------------------------ what a pass cannot do without

def work(case):
    kind, n = case["kind"], case.get("nrhs", 1)
    total_b = total_f = 0.0
    for d, kappa in _systems(case):
        V = math.prod(d)
        links, spinor, mom = 576.0 * V, 192.0 * V, 256.0 * V
        # CG iterations to 1e-11 (about 100 at kappa 0.12, 270 at 0.15, 540 at 0.155) grow towards the critical kappa
        iters = 50.0 / math.sqrt(max(0.005, 1.0 / kappa - 1.0 / 0.1585))
        op = 1368.0 * V
        if kind in ("static", "apply_mdagm"):
            b, f = links + 2 * spinor, 2 * op
        elif kind == "apply_m":
            b, f = links + 2 * spinor, op
        elif kind in ("solve", "batch", "uneven"):
            b, f = links + 2 * n * spinor, n * iters * (2 * op + 240.0 * V)
        elif kind == "autograd":
            b, f = 2 * links + 2 * spinor, 2 * iters * (2 * op + 240.0 * V)
        elif kind == "hmc":
            solves = case["steps"] + 2
            b, f = 2 * links + mom, solves * iters * (2 * op + 240.0 * V) + (solves - 1) * 20000.0 * V
        else:
            b, f = 2 * links + 3 * mom + spinor, 20000.0 * V
        total_b, total_f = total_b + b, total_f + f
    return {"bytes": total_b, "flops": total_f}


# ------------------------------------------------------------------ the same in plain 64-bit torch

# (gamma_mu psi)_s = sum_t G[mu][s][t] psi_t, DeGrand-Rossi basis
_GAMMA = [[[0, 0, 0, 1j], [0, 0, 1j, 0], [0, -1j, 0, 0], [-1j, 0, 0, 0]],
          [[0, 0, 0, -1], [0, 0, 1, 0], [0, 1, 0, 0], [-1, 0, 0, 0]],
          [[0, 0, 1j, 0], [0, 0, 0, -1j], [-1j, 0, 0, 0], [0, 1j, 0, 0]],
          [[0, 0, 1, 0], [0, 0, 0, 1], [1, 0, 0, 0], [0, 1, 0, 0]]]


def _spin(mu, sign, psi):
    """(1 + sign gamma_mu) psi."""
    out = []
    for s in range(4):
        v = psi[:, s]
        for t in range(4):
            if _GAMMA[mu][s][t]:
                v = v + sign * _GAMMA[mu][s][t] * psi[:, t]
        out.append(v)
    return torch.stack(out, 1)


def _shift(f, dims, mu, step):
    """Field at x + step mu."""
    g = f.view(dims[3], dims[2], dims[1], dims[0], *f.shape[1:])
    return torch.roll(g, -step, dims=3 - mu).reshape(f.shape)


def _color(U, psi):
    return (U[:, None] * psi[:, :, None]).sum(-1)


def _M(U, psi, dims, kappa, dagger=False):
    V = psi.shape[0]
    t = torch.arange(V, device=psi.device) // (dims[0] * dims[1] * dims[2])
    hop = torch.zeros_like(psi)
    for mu in range(4):
        sf = 1.0 if dagger else -1.0
        fwd = _color(U[:, mu], _shift(_spin(mu, sf, psi), dims, mu, 1))
        bwd = _shift(_color(U[:, mu].conj().transpose(1, 2), _spin(mu, -sf, psi)), dims, mu, -1)
        if mu == 3:
            fwd = torch.where((t == dims[3] - 1)[:, None, None], -fwd, fwd)
            bwd = torch.where((t == 0)[:, None, None], -bwd, bwd)
        hop = hop + fwd + bwd
    return psi - kappa * hop


def _MdagM(U, psi, dims, kappa):
    return _M(U, _M(U, psi, dims, kappa), dims, kappa, True)


def _solve(U, phi, dims, kappa, tol=1e-13):
    x, r = torch.zeros_like(phi), phi.clone()
    p, rr = r.clone(), float(torch.linalg.vector_norm(phi)) ** 2
    stop = tol * tol * rr
    for _ in range(5000):
        if rr <= stop:
            break
        Ap = _MdagM(U, p, dims, kappa)
        a = rr / torch.sum(p.conj() * Ap).real.item()
        x, r = x + a * p, r - a * Ap
        new = float(torch.linalg.vector_norm(r)) ** 2
        p, rr = r + (new / rr) * p, new
    return x


def _generators():
    z = torch.zeros((8, 3, 3), dtype=torch.complex128)
    for a, (i, j) in ((0, (0, 1)), (3, (0, 2)), (5, (1, 2))):
        z[a, i, j] = z[a, j, i] = 1
        z[a + 1, i, j], z[a + 1, j, i] = -1j, 1j
    z[2, 0, 0], z[2, 1, 1] = 1, -1
    z[7] = torch.diag(torch.tensor([1, 1, -2], dtype=torch.complex128)) / 3 ** 0.5
    return (z / 2 ** 0.5).to(DEV)


def _force(G, U):
    """d S / d w of U -> exp(i w t_a) U from the complex gradient G."""
    T = _generators()
    W = U @ G.conj().transpose(-1, -2)          # Re tr(i t_a U G^dag) = - Im tr(t_a U G^dag)
    return -torch.einsum("aij,vmji->vma", T, W).imag


def _gauge_action(U, dims, beta):
    S = 0.0
    for mu in range(4):
        for nu in range(mu + 1, 4):
            P = U[:, mu] @ _shift(U[:, nu], dims, mu, 1) @ _shift(U[:, mu], dims, nu, 1).conj().transpose(1, 2) \
                @ U[:, nu].conj().transpose(1, 2)
            S = S + beta * (1 - torch.diagonal(P, dim1=1, dim2=2).sum(1).real / 3).sum()
    return S


def _fermion_gradient(U, X, dims, kappa):
    """Complex gradient of phi^dag (M^dag M)^-1 phi at fixed X: that of -2 Re <Y, M(U) X>, Y = M X."""
    Y = _M(U, X, dims, kappa)
    Ua = U.clone().requires_grad_(True)
    f = -2 * torch.sum(Y.conj() * _M(Ua, X, dims, kappa)).real
    return torch.autograd.grad(f, Ua)[0]


def exact(case, seed):
    kind, kappa, dims = case["kind"], case["kappa"], _dims(case)
    V = sum(math.prod(d) for d, _ in _systems(case)) * case.get("nrhs", 1)
    if kind == "hmc" or (kind in ("solve", "batch", "uneven", "autograd") and V > 150000):
        return None
    s = prepare(case, seed)
    U, phi = s.U[0], s.phi[0]
    if kind in ("static", "apply_mdagm"):
        return _MdagM(U, phi, dims, kappa)
    if kind == "apply_m":
        return _M(U, phi, dims, kappa, case["dagger"])
    if kind == "solve":
        return _solve(U, phi, dims, kappa)
    if kind == "batch":
        return [torch.stack([_solve(U, p, dims, kappa) for p in phi])]
    if kind == "uneven":
        return [_solve(u, p, d, k) for u, p, (d, k) in zip(s.U, s.phi, _systems(case))]
    if kind == "autograd":
        X = _solve(U, phi, dims, kappa)
        return {"S": torch.sum(phi.conj() * X).real, "dU": _fermion_gradient(U, X, dims, kappa), "dphi": 2 * X}
    Ua = U.clone().requires_grad_(True)
    S = _gauge_action(Ua, dims, case["beta"])
    G = torch.autograd.grad(S, Ua)[0]
    P = torch.einsum("vma,aij->vmij", s.p.to(torch.complex128), _generators())
    return {"F": _force(G, U), "Ff": _force(_fermion_gradient(U, phi, dims, kappa), U),
            "U": torch.matrix_exp(0.05j * P) @ U, "action": float(S.detach())}

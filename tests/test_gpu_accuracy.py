"""FP64 entry points computed in fixed point (csrc/lq_fix64.cuh, lq_fixsu3.cuh) against extended precision,
on the inputs where a fixed unit could cost digits that FP64 arithmetic keeps."""
import numpy as np
import pytest

from oracle.wilson import apply_M
from synth import Lattice, gauge_exp_iA, source
from tests.gpu_common import require_gpu, dev, host, torch

pytestmark = pytest.mark.gpu
EPS = 2.0 ** -53


@pytest.fixture(scope="module")
def lq():
    return require_gpu()


class _Context:
    def __init__(self, lq, dims, U):
        self.lq, self.dims, self.U = lq, dims, U

    def __enter__(self):
        self.ctx = self.lq.lq_create(self.dims)
        self.lq.lq_gauge_set(self.ctx, dev(self.U))
        return self.ctx

    def __exit__(self, *exc):
        self.lq.lq_destroy(self.ctx)


def _M(lq, ctx, psi, kappa, dagger=False):
    out = torch.empty(psi.shape, dtype=torch.complex128, device="cuda")
    lq.lq_apply_M(ctx, out, dev(psi), kappa, dagger, lq.LQ_F64)
    return host(out)


def _gauge_force(lq, ctx, V, beta):
    F = torch.empty((V, 4, 8), dtype=torch.float64, device="cuda")
    lq.lq_gauge_force(ctx, F, beta)
    return host(F)


def _fermion_force(lq, ctx, X, kappa):
    F = torch.empty((X.shape[0], 4, 8), dtype=torch.float64, device="cuda")
    lq.lq_fermion_force(ctx, F, dev(X), kappa)
    return host(F)


# ------------------------------------------------------------ short links
@pytest.mark.parametrize("scale", [0.3, 0.1, 1e-2, 1e-4, 1e-8])
@pytest.mark.parametrize("dims", [(4, 4, 4, 4), (3, 5, 2, 7)])
def test_short_links(lq, dims, scale):
    """Links that are a multiple of unitary ones, shorter than 1: every result to FP64 accuracy relative to
    its own powers of the scale.  Bounds as for unitary links (128 units of 2^-53 of the largest product for
    plaquette and gauge force, 64 for the operator, 64 * 24 for the fermion force) times those powers."""
    from oracle.fermion import fermion_force_from_X
    from oracle.gauge import gauge_force, plaquette
    lat = Lattice(dims)
    U, psi, beta = scale * gauge_exp_iA(lat, 0.3, 6), source(lat, 6), 5.6
    kappa = 0.15 / scale
    with _Context(lq, dims, U) as ctx:
        P = lq.lq_plaquette(ctx)
        F = _gauge_force(lq, ctx, lat.V, beta)
        m = _M(lq, ctx, psi, kappa)
        Ff = _fermion_force(lq, ctx, psi, kappa)
    out = torch.empty(psi.shape, dtype=torch.complex128, device="cuda")
    lq.lq_apply_MdagM_static(out, dev(U), dev(psi), dims, kappa)
    s4 = scale ** 4
    assert abs(P - plaquette(U, dims)) <= 128 * EPS * 3 * s4
    assert np.abs(F - gauge_force(U, dims, beta)).max() <= 128 * EPS * beta / 3 * 18 * s4
    top = np.abs(psi).max()
    Y = apply_M(U, psi, dims, kappa)
    assert np.abs(m - Y).max() <= 64 * EPS * top
    ref = fermion_force_from_X(U, psi, dims, kappa)
    assert np.abs(Ff - ref).max() <= 64 * 24 * EPS * 0.3 * top * np.abs(Y).max()
    grow = 1 + 8 * 0.15 * 3
    assert np.abs(host(out) - apply_M(U, Y, dims, kappa, True, True)).max() <= 64 * EPS * grow ** 2 * top


def test_open_boundary_with_a_field_that_falls(lq):
    """Temporal links of zero across the boundary and a field 1e-14 times smaller per time slice: a site next to
    the boundary owes nothing to the large values behind the zero link.  Bound: 64 units of 2^-53 of the
    largest component among the site and the neighbours it has a link to (all four last slices are compared)."""
    dims = (4, 3, 4, 6)
    lat = Lattice(dims)
    U, psi = gauge_exp_iA(lat, 0.3, 6), source(lat, 6)
    x = lat.coords()
    t = x[:, 3]
    U[t == dims[3] - 1, 3] = 0.0
    psi = psi * (1e-14 ** t)[:, None, None]
    with _Context(lq, dims, U) as ctx:
        got = _M(lq, ctx, psi, 0.15)
    out = torch.empty(psi.shape, dtype=torch.complex128, device="cuda")
    lq.lq_apply_MdagM_static(out, dev(U), dev(psi), dims, 0.15)
    ref = apply_M(U, psi, dims, 0.15)
    top = np.array([np.abs(psi[t == k]).max() for k in range(dims[3])])
    for k in range(dims[3]):
        tol = 64 * EPS * max(top[k], top[k - 1] if k > 0 else 0.0)
        assert np.abs(got - ref)[t == k].max() <= tol, k
    ref = apply_M(U, ref, dims, 0.15, True, True)
    for k in range(dims[3]):
        tol = 64 * EPS * (1 + 8 * 0.15 * 3) ** 2 * max(top[j] for j in range(max(0, k - 2), dims[3]))
        assert np.abs(host(out) - ref)[t == k].max() <= tol, k


# ------------------------------------------------------------ extended precision
# numpy's long double (64 bits of mantissa or more on the machines this runs on); matrices by explicit sums.
LD, CLD = np.longdouble, np.clongdouble


def _generators():
    T = np.zeros((8, 3, 3), CLD)
    for a, (i, j) in ((0, (0, 1)), (3, (0, 2)), (5, (1, 2))):
        T[a, i, j] = T[a, j, i] = 1
        T[a + 1, i, j], T[a + 1, j, i] = -1j, 1j
    T[2, 0, 0], T[2, 1, 1] = 1, -1
    T[7] = np.diag([1, 1, -2]).astype(CLD) / np.sqrt(LD(3))
    return T / np.sqrt(LD(2))


def _mm(a, b):
    return (a[..., :, :, None] * b[..., None, :, :]).sum(-2)


def _dag(a):
    return a.conj().swapaxes(-1, -2)


def _rms_rel(F, ref):
    """Root mean square over the links of |F - ref| / |ref| (2-norms of the eight components)."""
    d = np.sqrt(((F.astype(LD) - ref) ** 2).sum(-1) / (ref ** 2).sum(-1))
    return float(np.sqrt((d ** 2).mean()))


def _ld_M(U, psi, dims, kappa):
    from oracle.conventions import GAMMA, neighbours
    fwd, bwd, sf, sb = neighbours(dims)
    out = psi.copy()
    for mu in range(4):
        g = GAMMA[mu].astype(CLD)
        for f, n, u, sg in ((sf, fwd, U[:, mu], -1), (sb, bwd, _dag(U[bwd[mu], mu]), 1)):
            p = psi[n[mu]]
            p = p + sg * _mm(np.broadcast_to(g, (len(p), 4, 4)), p)
            out = out - LD(kappa) * f[mu][:, None, None] * _mm(p, u.swapaxes(-1, -2))
    return out


def _ld_fermion_force(U, X, dims, kappa):
    """F_a = 2 kappa s Re[i Y(x)^dag (1 - g) t_a U X(x+mu) - i Y(x+mu)^dag (1 + g) U^dag t_a X(x)]."""
    from oracle.conventions import GAMMA, neighbours
    fwd, _, sf, _ = neighbours(dims)
    U, X, T = U.astype(CLD), X.astype(CLD), _generators()
    Y = _ld_M(U, X, dims, kappa)
    F = np.zeros((len(X), 4, 8), LD)
    for mu in range(4):
        g = np.broadcast_to(GAMMA[mu].astype(CLD), (len(X), 4, 4))
        Xf, Yf = X[fwd[mu]], Y[fwd[mu]]
        a = _mm(Xf, U[:, mu].swapaxes(-1, -2))                         # U X(x+mu)
        b = _mm(Yf + _mm(g, Yf), U[:, mu].swapaxes(-1, -2))            # U (1 + g) Y(x+mu)
        C = _mm(a.swapaxes(-1, -2), (Y - _mm(g, Y)).conj()) - _mm(X.swapaxes(-1, -2), b.conj())
        tr = (T[None] * C[:, None].swapaxes(-1, -2)).sum((-1, -2))     # sum_ij T_ij C_ji
        F[:, mu] = LD(2) * LD(kappa) * sf[mu][:, None] * (1j * tr).real
    return F


@pytest.mark.parametrize("fall", [1.0, 2.0, 8.0, 1024.0])
@pytest.mark.parametrize("dims", [(4, 4, 4, 6), (3, 5, 2, 7), (8, 6, 5, 9)])
def test_fermion_force_of_a_falling_field(lq, dims, fall):
    """X a factor smaller on every time slice (a propagator away from its source): no link's force is further
    from extended precision than FP64 arithmetic in the order of the oracle, root mean square over the
    links of each direction.  (Temporal links into and across the boundary, and those of the steepest fall, are
    left out: there Y comes from one large neighbour whose part the projection takes away again, and what
    is left are the roundings of Y to FP64, the same in any arithmetic.)"""
    from oracle.fermion import fermion_force_from_X
    lat = Lattice(dims)
    U, X = gauge_exp_iA(lat, 0.3, 6), source(lat, 6)
    X = X * (fall ** -lat.coords()[:, 3].astype(float))[:, None, None]
    ref = _ld_fermion_force(U, X, dims, 0.15)
    plain = fermion_force_from_X(U, X, dims, 0.15)
    with _Context(lq, dims, U) as ctx:
        F = _fermion_force(lq, ctx, X, 0.15)
    for mu in range(4 if fall < 100 else 3):
        sel = lat.coords()[:, 3] < dims[3] - 2 * (mu == 3)
        assert _rms_rel(F[sel, mu], ref[sel, mu]) <= _rms_rel(plain[sel, mu], ref[sel, mu]), mu


def _ld_gauge_force(U, dims, beta):
    from oracle.conventions import neighbours
    fwd, bwd, _, _ = neighbours(dims, False)
    U = U.astype(CLD)
    T, F = _generators(), np.zeros((len(U), 4, 8), LD)
    for mu in range(4):
        S = np.zeros((len(U), 3, 3), CLD)
        for nu in range(4):
            if nu != mu:
                xm, xn, xb = fwd[mu], fwd[nu], bwd[nu]
                S += _mm(_mm(U[xm, nu], _dag(U[xn, mu])), _dag(U[:, nu]))
                S += _mm(_mm(_dag(U[xb[xm], nu]), _dag(U[xb, mu])), U[xb, nu])
        W = _mm(U[:, mu], S)
        F[:, mu] = LD(beta) / 3 * (T[None] * W[:, None].swapaxes(-1, -2)).sum((-1, -2)).imag
    return F


@pytest.mark.parametrize("rough", [0.3, 0.05, 1e-2, 3e-3, 1e-3, 1e-4, 1e-6, "half"])
@pytest.mark.parametrize("dims", [(4, 4, 4, 4), (3, 5, 2, 7), (8, 6, 5, 9)])
def test_gauge_force_of_smooth_links(lq, dims, rough):
    """Links close to 1, where the force is as small as their roughness and FP64 products keep its relative
    accuracy: no further from extended precision than FP64 arithmetic in the order of the oracle (root mean
    square over the links; 1.25: the spread of that figure over some hundred links).  "half": smooth on one
    half of the time slices, rough on the other, each half of the links compared by itself."""
    from oracle.gauge import gauge_force
    lat = Lattice(dims)
    U = gauge_exp_iA(lat, 0.3 if rough == "half" else rough, 6)
    part = np.zeros(lat.V, bool)
    if rough == "half":
        t = lat.coords()[:, 3]
        U[t < dims[3] // 2] = gauge_exp_iA(lat, 1e-5, 7)[t < dims[3] // 2]
        part = (t > 0) & (t < dims[3] // 2 - 1)
    ref, plain = _ld_gauge_force(U, dims, 5.6), gauge_force(U, dims, 5.6)
    with _Context(lq, dims, U) as ctx:
        F = _gauge_force(lq, ctx, lat.V, 5.6)
    for sel in (part, ~part):
        if sel.any():
            assert _rms_rel(F[sel], ref[sel]) <= 1.25 * _rms_rel(plain[sel], ref[sel])


# ------------------------------------------------------------ fields with zero spins
def _projected(psi, keep):
    out = np.zeros_like(psi)
    out[:, keep] = psi[:, keep]
    return out


@pytest.mark.parametrize("keep", [[0, 1], [2, 3], [1], [0, 2, 3]])
@pytest.mark.parametrize("dims", [(4, 4, 4, 4), (3, 5, 2, 7), (16, 12, 12, 18)])
def test_operator_on_fields_with_zero_spins(lq, dims, keep):
    """Chirally projected and spin-diluted fields; bound as for full fields, 64 units of 2^-53 of the largest
    component near, and exact zeros stay zero."""
    lat = Lattice(dims)
    U, psi = gauge_exp_iA(lat, 0.3, 6), _projected(source(lat, 6), keep)
    with _Context(lq, dims, U) as ctx:
        for dagger in (False, True):
            got, ref = _M(lq, ctx, psi, 0.15, dagger), apply_M(U, psi, dims, 0.15, True, dagger)
            assert np.abs(got - ref).max() <= 64 * EPS * np.abs(psi).max()
            assert np.all(got[ref == 0] == 0)


def test_zero_spins_cost_no_more_than_full_fields(lq):
    """A spin that is zero has no digits to lose, so a projected field takes the same path as a full one (FP64
    arithmetic at every site takes more than twice the time)."""
    dims = (24, 24, 24, 32)
    lat = Lattice(dims)
    gen = torch.Generator(device="cuda").manual_seed(3)
    psi = torch.randn((lat.V, 4, 3, 2), dtype=torch.float64, device="cuda", generator=gen)
    U = torch.eye(3, dtype=torch.complex128, device="cuda").repeat(lat.V, 4, 1, 1).contiguous()
    ctx = lq.lq_create(dims)
    try:
        lq.lq_gauge_set(ctx, U)
        full = torch.view_as_complex(psi)
        half = full.clone()
        half[:, 2:] = 0
        ms = [lq.lq_time_dslash(ctx, f, 0.15, False, lq.LQ_F64, 20) for f in (full, half)]
    finally:
        lq.lq_destroy(ctx)
    assert ms[1] <= 1.3 * ms[0], ms

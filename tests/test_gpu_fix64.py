"""The fixed-point FP64 operator (csrc/lq_fix64.cuh): the forms its rules send to different paths."""
import numpy as np
import pytest

from oracle.wilson import apply_M
from synth import Lattice, gauge_exp_iA, source
from tests.gpu_common import require_gpu, dev, host, torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lq():
    return require_gpu()


def _apply(lq, dims, U, psi, dagger, t_anti=True):
    ctx = lq.lq_create(dims, t_anti)
    try:
        lq.lq_gauge_set(ctx, dev(U))
        out = torch.empty(psi.shape, dtype=torch.complex128, device="cuda")
        lq.lq_apply_M(ctx, out, dev(psi), 0.15, dagger, lq.LQ_F64)
        return host(out)
    finally:
        lq.lq_destroy(ctx)


def _fields(dims, kind):
    """Spinors (and links) that reach one rule each."""
    lat = Lattice(dims)
    U, psi = gauge_exp_iA(lat, 0.3, 6), source(lat, 6)
    rng = np.random.default_rng(6)
    if kind == "site_range":            # neighbours of very different size: one exponent for eight of them
        psi = psi * np.exp(rng.normal(0, 12, (lat.V, 1, 1)))
    elif kind == "spin_range":          # spins more than 2^6 apart: FP64 arithmetic
        psi[::3, 1] *= 1e-7
    elif kind == "point":               # one non-zero component
        psi = np.zeros_like(psi)
        psi[lat.V // 2, 2, 1] = 1.0 - 2.0j
    elif kind == "tiny":                # below the smallest exponent the fixed-point path takes
        psi = psi * 2.0 ** -1000
    elif kind == "huge":
        psi = psi * 2.0 ** 1000
    elif kind == "ones":                # limb edges: links of exactly 1, powers of two
        U = np.tile(np.eye(3, dtype=np.complex128), (lat.V, 4, 1, 1))
        psi = np.sign(psi.real) + 1j * np.sign(psi.imag)
    elif kind == "not_unitary":         # general matrices: FP64 arithmetic at every site
        U = U * (1.5 + 0.1 * rng.normal(size=(lat.V, 4, 1, 1)))
    return U, psi


@pytest.mark.parametrize("dims", [(4, 4, 4, 4), (3, 5, 2, 7), (16, 12, 12, 18)])
@pytest.mark.parametrize("kind", ["gauss", "site_range", "spin_range", "point", "tiny", "huge", "ones", "not_unitary"])
@pytest.mark.parametrize("dagger", [False, True])
def test_matches_oracle_element_by_element(lq, dims, kind, dagger):
    """(16, 12, 12, 18) has more blocks than SMs (the capped kernel), the others fewer.  Bound per
    element: 8 hops, each rounding FP64 products and sums of the components one site reads, at most
    64 units of 2^-53 of the largest of them (the fixed-point path keeps 2^-56 of it), times the
    largest link element."""
    U, psi = _fields(dims, kind)
    scale = 1.0
    if kind in ("tiny", "huge"):        # the oracle's own sums at a scale without underflow
        scale = 2.0 ** (-1000 if kind == "tiny" else 1000)
    ref = apply_M(U, psi / scale, dims, 0.15, True, dagger)
    got = _apply(lq, dims, U, psi, dagger) / scale
    lat = Lattice(dims)
    a = np.abs(psi / scale).max(axis=(1, 2)).reshape(dims[::-1])
    near = a.copy()
    for ax in range(4):
        near = np.maximum(near, np.maximum(np.roll(a, 1, ax), np.roll(a, -1, ax)))
    tol = 64 * 2.0 ** -53 * max(1.0, np.abs(U).max()) * near.reshape(lat.V, 1, 1)
    assert np.all(np.abs(got - ref) <= tol)
    assert np.all(got[ref == 0] == 0)


@pytest.mark.parametrize("value", [np.nan, np.inf])
def test_non_finite_values_reach_their_neighbours_only(lq, value):
    dims = (4, 6, 4, 4)
    lat = Lattice(dims)
    U, psi = gauge_exp_iA(lat, 0.3, 6), source(lat, 6)
    s = 77
    psi[s, 0, 0] = value
    got = _apply(lq, dims, U, psi, False)
    finite = np.isfinite(got).all(axis=(1, 2))
    x = lat.coords()
    d = np.abs(x - x[s])
    d = np.minimum(d, np.array(dims) - d).sum(axis=1)
    assert np.array_equal(finite, d > 1)


@pytest.mark.parametrize("dims", [(4, 4, 4, 4), (3, 5, 2, 7), (2, 2, 2, 2)])
@pytest.mark.parametrize("kind", ["gauss", "ones", "not_unitary"])
def test_plaquette_and_gauge_force(lq, dims, kind):
    """Staples and plaquettes in fixed point, and in FP64 arithmetic for general matrices, against
    the oracle.  Bounds: a staple is three FP64 matrix products (at most 3 * 9 roundings of sums of
    |U|^3), six of them times a link; 128 units of 2^-53 of (beta / 3) * 18 * max |U|^4."""
    from oracle.gauge import gauge_force, plaquette
    U, _ = _fields(dims, kind)
    V = Lattice(dims).V
    ctx = lq.lq_create(dims)
    try:
        lq.lq_gauge_set(ctx, dev(U))
        F = torch.empty((V, 4, 8), dtype=torch.float64, device="cuda")
        lq.lq_gauge_force(ctx, F, 5.6)
        F, P = host(F), lq.lq_plaquette(ctx)
    finally:
        lq.lq_destroy(ctx)
    top = max(1.0, np.abs(U).max()) ** 4
    unit = 128 * 2.0 ** -53
    assert np.abs(F - gauge_force(U, dims, 5.6)).max() <= unit * 5.6 / 3 * 18 * top
    assert abs(P - plaquette(U, dims)) <= unit * 3 * top


@pytest.mark.parametrize("eps", [1e-9, 0.02, 0.08, 0.3, 0.45, 2.0])
def test_link_update_over_step_sizes(lq, eps):
    """exp(i eps P) U by 12 or 18 terms of its series or by the closed form, per link by the size of
    eps P (the steps straddle both limits), momenta of zero among them.  Bound: 64 units of 2^-53
    (about 40 rounded sums of numbers of order 1; the closed form's sines of arguments of order eps |p|)."""
    from oracle.su3 import link_update
    dims = (4, 3, 2, 5)
    lat = Lattice(dims)
    U = gauge_exp_iA(lat, 0.3, 6)
    p = np.random.default_rng(3).normal(size=(lat.V, 4, 8))
    p[5] = 0.0
    ctx = lq.lq_create(dims)
    try:
        lq.lq_gauge_set(ctx, dev(U))
        lq.lq_link_update(ctx, dev(p), eps)
        got = torch.empty(U.shape, dtype=torch.complex128, device="cuda")
        lq.lq_gauge_get(ctx, got)
    finally:
        lq.lq_destroy(ctx)
    got = host(got)
    ref = link_update(U, p, eps)
    assert np.abs(got - ref).max() <= 64 * 2.0 ** -53 * max(1.0, eps)
    assert np.abs(got @ got.conj().swapaxes(-1, -2) - np.eye(3)).max() <= 16 * 2.0 ** -53


@pytest.mark.parametrize("dims", [(4, 4, 4, 4), (3, 5, 2, 7), (2, 2, 2, 2)])
@pytest.mark.parametrize("kind", ["gauss", "site_range", "spin_range", "point", "huge", "not_unitary"])
def test_fermion_force(lq, dims, kind):
    """Force of X and Y = M X in fixed point and, where their exponents or the links do not fit, in
    FP64.  Bound per link: two outer products of projected spinors (rounded products of U, X and Y,
    at most 64 roundings) of the largest |X| and |Y| of its two sites, times 2 kappa max |U|."""
    from oracle.fermion import fermion_force_from_X
    U, X = _fields(dims, kind)
    scale = 2.0 ** 500 if kind == "huge" else 1.0      # X^2 has to stay finite
    X = X / (2.0 ** 500 if kind == "huge" else 1.0)
    V = Lattice(dims).V
    ctx = lq.lq_create(dims)
    try:
        lq.lq_gauge_set(ctx, dev(U))
        F = torch.empty((V, 4, 8), dtype=torch.float64, device="cuda")
        lq.lq_fermion_force(ctx, F, dev(X), 0.15)
        F = host(F) / scale / scale
    finally:
        lq.lq_destroy(ctx)
    X = X / scale
    ref = fermion_force_from_X(U, X, dims, 0.15)
    Y = apply_M(U, X, dims, 0.15)
    grid = dims[::-1]
    ax, ay = (np.abs(f).max(axis=(1, 2)).reshape(grid) for f in (X, Y))
    # Y itself is rounded relative to the sites M reads
    ny = np.maximum(ay, ax)
    for m in range(4):
        ny = np.maximum(ny, np.maximum(np.roll(ax, 1, m), np.roll(ax, -1, m)))
    u = max(1.0, np.abs(U).max()) ** 2
    for mu in range(4):
        fwd = lambda a: np.maximum(a, np.roll(a, -1, 3 - mu))   # noqa: E731
        tol = 2.0 ** -53 * 64 * 24 * 0.3 * u * (fwd(ax) * fwd(ny)).reshape(V, 1)
        assert np.all(np.abs(F[:, mu] - ref[:, mu]) <= tol), mu


@pytest.mark.parametrize("dims", [(4, 4, 4, 4), (3, 5, 2, 7), (16, 12, 12, 18)])
@pytest.mark.parametrize("kind", ["gauss", "site_range", "spin_range", "point", "ones", "not_unitary", "one_bad_link"])
def test_static_mdagm(lq, dims, kind):
    """M^dag M on canonical buffers against the oracle; one bad link sends only the sites that read
    it to FP64 arithmetic.  Bound per element: as above for both applications, 64 units of 2^-53 of
    the largest component within two steps, times (1 + 8 * 0.15 * 3 max |U|)^2."""
    U, psi = _fields(dims, "gauss" if kind == "one_bad_link" else kind)
    lat = Lattice(dims)
    if kind == "one_bad_link":
        U[lat.V // 3, 2] *= 3.0
    out = torch.empty(psi.shape, dtype=torch.complex128, device="cuda")
    lq.lq_apply_MdagM_static(out, dev(U), dev(psi), dims, 0.15)
    ref = apply_M(U, apply_M(U, psi, dims, 0.15), dims, 0.15, True, True)
    near = np.abs(psi).max(axis=(1, 2)).reshape(dims[::-1])
    for _ in range(2):
        a = near
        for ax in range(4):
            near = np.maximum(near, np.maximum(np.roll(a, 1, ax), np.roll(a, -1, ax)))
    grow = 1 + 8 * 0.15 * 3 * max(1.0, np.abs(U).max())
    tol = 64 * 2.0 ** -53 * grow ** 2 * near.reshape(lat.V, 1, 1)
    assert np.all(np.abs(host(out) - ref) <= tol)

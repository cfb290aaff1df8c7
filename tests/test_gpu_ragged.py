"""Solves inside one cluster (csrc/k_cgcluster.cu) on lattices that end in the middle of a warp."""
import numpy as np
import pytest

from oracle.cg import cg_MdagM
from synth import Lattice, gauge_exp_iA, source
from tests.gpu_common import require_gpu, dev, host, rel_err, torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lq():
    return require_gpu()


# 27 + 3 lanes of one warp; 625 = 15 x 40 + 25 over blocks of 64; 2401 over blocks of 160; 5831 over blocks of 384
@pytest.mark.parametrize("dims", [(3, 5, 2, 2), (5, 5, 5, 5), (7, 7, 7, 7), (7, 7, 7, 17)])
@pytest.mark.parametrize("prec", ["f32_12", "f16_12", "bf16_12"])
def test_ragged_lattices(lq, dims, prec):
    """The barrier is entered after loops that only some lanes of the last warp run.  Two solutions at a true
    residual of 1e-11 differ by at most cond(M^dag M) ~ 1e3 times their sum (kappa 0.14)."""
    lat = Lattice(dims)
    U, phi = gauge_exp_iA(lat, 0.3, 11), source(lat, 11)
    ref = cg_MdagM(U, phi, dims, 0.14, 1e-13)[0]
    ctx = lq.lq_create(dims)
    try:
        lq.lq_gauge_set(ctx, dev(U))
        x = torch.zeros(phi.shape, dtype=torch.complex128, device="cuda")
        status, st = lq.lq_solve_MdagM(ctx, x, dev(phi), 0.14, 1e-11, 3000, lq.PRECISIONS[prec], 30)
        assert status == lq.LQ_OK and st["true_rel_resid"] <= 1e-11
        assert rel_err(host(x), ref) < 2e-8
    finally:
        lq.lq_destroy(ctx)
    assert np.isfinite(host(x)).all()


@pytest.mark.parametrize("dims", [(4, 4, 4, 4), (8, 8, 8, 20)])
def test_links_replaced_before_overlapped_launches(lq, dims):
    """New links and a call whose first stencil launch may be set up while its predecessor still runs, over and
    over: every result is, to the bit, that of a context that only ever held those links."""
    lat = Lattice(dims)
    Us = [dev(gauge_exp_iA(lat, 0.3, s)) for s in (1, 2)]
    phi = dev(source(lat, 3))

    def results(ctx):
        F = torch.empty((lat.V, 4, 8), dtype=torch.float64, device="cuda")
        m, x = torch.empty_like(phi), torch.zeros_like(phi)
        lq.lq_fermion_force(ctx, F, phi, 0.14)
        lq.lq_apply_MdagM(ctx, m, phi, 0.14, lq.LQ_F64)
        lq.lq_solve_MdagM(ctx, x, phi, 0.14, 1e-10, 60, lq.LQ_F32_12, 20)
        return [host(v).copy() for v in (F, m, x)]

    want = []
    for U in Us:
        ctx = lq.lq_create(dims)
        lq.lq_gauge_set(ctx, U)
        want.append(results(ctx))
        lq.lq_destroy(ctx)
    ctx = lq.lq_create(dims)
    try:
        for i in range(20):
            lq.lq_gauge_set(ctx, Us[i & 1])
            for got, ref in zip(results(ctx), want[i & 1]):
                assert np.array_equal(got, ref)
    finally:
        lq.lq_destroy(ctx)

"""Calls that meet the end of device memory: an error or the same result, and a context that works afterwards."""
import numpy as np
import pytest

from synth import Lattice, gauge_exp_iA, source
from tests.gpu_common import require_gpu, dev, host, torch

pytestmark = pytest.mark.gpu
DIMS = (16, 16, 16, 32)            # an FP64 spinor field is 24 MiB (+ 0.5 of exponent words), fixed-point links are 72
MIB = 1 << 20


@pytest.fixture(scope="module")
def lq():
    return require_gpu()


class _Full:
    """Device memory filled up to `leave` bytes, in the caching allocator's 2 MiB steps."""

    def __init__(self, leave):
        self.leave = leave

    def __enter__(self):
        torch.cuda.synchronize()
        torch.cuda.empty_cache()
        self.blocks = []
        for _ in range(64):
            n = (torch.cuda.mem_get_info()[0] - self.leave) // (2 * MIB) * (2 * MIB)
            if n <= 0:
                break
            try:
                self.blocks.append(torch.empty(n, dtype=torch.uint8, device="cuda"))
            except torch.cuda.OutOfMemoryError:
                self.leave += 2 * MIB

    def __exit__(self, *exc):
        self.blocks = None
        torch.cuda.synchronize()
        torch.cuda.empty_cache()


@pytest.fixture(scope="module")
def fields():
    lat = Lattice(DIMS)
    return dev(gauge_exp_iA(lat, 0.3, 6)), dev(source(lat, 6))


@pytest.mark.parametrize("leave", [100, 190, 194, 196, 198, 200, 386, 390, 394, 400])
@pytest.mark.parametrize("prec", ["f64", "f16_12"])
def test_a_field_that_does_not_fit(lq, leave, prec):
    """A spinor field of FP64 or 16-bit storage is two allocations (192 or 48 MiB and 4 MiB here); when only the
    first fits, the call fails and the field is not taken for complete by the next one."""
    dims = (32, 32, 32, 32)
    V, p = 32 ** 4, lq.PRECISIONS[prec]
    gen = torch.Generator(device="cuda").manual_seed(3)
    psi = torch.view_as_complex(torch.randn((V, 4, 3, 2), dtype=torch.float64, device="cuda", generator=gen))
    U = torch.eye(3, dtype=torch.complex128, device="cuda").repeat(V, 4, 1, 1).contiguous()
    want, out = torch.empty_like(psi), torch.empty_like(psi)
    ctx = lq.lq_create(dims)
    lq.lq_gauge_set(ctx, U)
    lq.lq_apply_M(ctx, want, psi, 0.12, False, p)          # also loads the kernels
    lq.lq_destroy(ctx)
    ctx = lq.lq_create(dims)
    try:
        lq.lq_gauge_set(ctx, U)
        lq.lq_plaquette(ctx)
        del U
        with _Full((leave + (0 if prec == "f64" else 96 + 48 - 192)) * MIB):
            try:
                lq.lq_apply_M(ctx, out, psi, 0.12, False, p)
                torch.cuda.synchronize()
            except lq.LQError as e:
                assert e.status == lq.LQ_ERR_CUDA
        lq.lq_apply_M(ctx, out, psi, 0.12, False, p)
        assert torch.equal(out, want)
    finally:
        lq.lq_destroy(ctx)


def test_links_that_fit_only_once(lq, fields):
    """The fixed-point copy of the links is an aid: without memory for it every call that needs none itself still
    answers, in FP64 arithmetic.  Bounds: 64 units of 2^-53 of the largest component (operator, sums of at most
    64 rounded products), 128 * 18 units of beta / 3 (gauge force), 128 * 3 (plaquette)."""
    U, psi = fields
    kappa, beta, eps = 0.15, 5.6, 2.0 ** -53
    V = psi.shape[0]
    want, got = [], []
    for leave, res in ((None, want), (64 * MIB, got)):
        ctx = lq.lq_create(DIMS)
        try:
            F, p = (torch.zeros((V, 4, 8), dtype=torch.float64, device="cuda") for _ in range(2))
            out = torch.empty_like(psi)
            lq.lq_gauge_set(ctx, U)
            lq.lq_link_update(ctx, p, 0.1)          # allocates the momentum fields; exp(0) U
            lq.lq_gauge_set(ctx, U)

            def calls():
                res.append(lq.lq_plaquette(ctx))
                lq.lq_gauge_force(ctx, F, beta)
                res.append(host(F).copy())
                lq.lq_fermion_force(ctx, F, psi, kappa)
                res.append(host(F).copy())
                lq.lq_apply_M(ctx, out, psi, kappa, False, lq.LQ_F64)
                res.append(host(out).copy())

            if leave is None:
                calls()
            else:
                with _Full(leave):
                    calls()
                calls()                             # and after memory is there again
        finally:
            lq.lq_destroy(ctx)
    top = float(torch.abs(psi).max())
    tol = [128 * 3 * eps, 128 * 18 * eps * beta / 3, 64 * 24 * eps * 0.3 * top * 4 * top, 64 * eps * top]
    for k, g in enumerate(got):
        assert np.abs(g - want[k % 4]).max() <= tol[k % 4], k
    x = torch.zeros_like(psi)
    ctx = lq.lq_create(DIMS)
    try:
        lq.lq_gauge_set(ctx, U)
        with _Full(64 * MIB):
            lq.lq_plaquette(ctx)
        for prec in (lq.LQ_F64, lq.LQ_F16_12):
            status, st = lq.lq_solve_MdagM(ctx, x, psi, 0.12, 1e-10, 2000, prec, 50)
            assert status == lq.LQ_OK and st["true_rel_resid"] <= 1e-10
        status, _, _, resid, _ = lq.lq_solve_batch([ctx], [x], [psi], [0.12], 1, 1e-10, 2000, lq.LQ_F16_12, 50)
        assert status == lq.LQ_OK and resid.max() <= 1e-10
    finally:
        lq.lq_destroy(ctx)

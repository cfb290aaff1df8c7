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


@pytest.mark.parametrize("leave", [8, 22, 24, 26, 28, 48, 50, 52])
@pytest.mark.parametrize("prec", ["f64", "f16_12"])
def test_a_field_that_does_not_fit(lq, fields, leave, prec):
    """A spinor field of 16-bit or FP64 storage is two allocations; when only the first fits, the call fails and
    the field is not taken for complete by the next one."""
    U, psi = fields
    p, out = lq.PRECISIONS[prec], torch.empty_like(psi)
    ctx = lq.lq_create(DIMS)
    try:
        lq.lq_gauge_set(ctx, U)
        lq.lq_plaquette(ctx)
        with _Full(leave * MIB):
            try:
                lq.lq_apply_M(ctx, out, psi, 0.15, False, p)
                torch.cuda.synchronize()
            except RuntimeError:
                pass
        lq.lq_apply_M(ctx, out, psi, 0.15, False, p)
        got = host(out).copy()
    finally:
        lq.lq_destroy(ctx)
    ctx = lq.lq_create(DIMS)
    try:
        lq.lq_gauge_set(ctx, U)
        lq.lq_apply_M(ctx, out, psi, 0.15, False, p)
        assert np.array_equal(got, host(out))
    finally:
        lq.lq_destroy(ctx)

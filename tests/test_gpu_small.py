"""Small lattices: CG iterations inside one cluster (csrc/k_cgcluster.cu), the FP64 operator split by
direction, and the sizes next to their limits."""
import functools

import numpy as np
import pytest

from oracle.cg import cg_MdagM
from synth import Lattice, gauge_exp_iA, source
from tests.gpu_common import require_gpu, dev, host, rel_err

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lq():
    return require_gpu()


@functools.lru_cache(maxsize=None)
def _system(dims):
    lat = Lattice(dims)
    U, phi = gauge_exp_iA(lat, 0.3, 11), source(lat, 11)
    return U, phi, cg_MdagM(U, phi, dims, 0.14, 1e-13)[0]


# one block, several blocks with a ragged last warp, all 16, the largest of the cluster, one beyond it;
# the largest of the split FP64 operator and one beyond
@pytest.mark.parametrize("dims", [(2, 2, 2, 2), (3, 5, 2, 7), (4, 4, 4, 8), (8, 8, 8, 12), (8, 8, 8, 13), (8, 8, 8, 16),
                                  (8, 8, 9, 16)])
@pytest.mark.parametrize("prec", ["f32", "f32_12", "f16_12", "bf16_12", "i16_12", "f64"])
def test_solves_around_the_limits(lq, dims, prec):
    """Every path stops on an FP64 residual of 1e-11; two such solutions differ by at most cond(M^dag M) ~
    1e3 times their sum (kappa 0.14).  The history has one entry per iteration, the last below the
    tolerance, and an iteration limit inside a chunk ends the solve there."""
    import torch
    U, phi, ref = _system(dims)
    ctx = lq.lq_create(dims)
    try:
        lq.lq_gauge_set(ctx, dev(U))
        x, p = torch.zeros(phi.shape, dtype=torch.complex128, device="cuda"), lq.PRECISIONS[prec]
        hist = np.zeros(3000)
        status, st = lq.lq_solve_MdagM(ctx, x, dev(phi), 0.14, 1e-11, 3000, p, 30, hist=hist)
        assert status == lq.LQ_OK and st["true_rel_resid"] <= 1e-11
        assert rel_err(host(x), ref) < 2e-8
        n = st["iterations"]
        assert np.all(hist[:n] > 0) and hist[n - 1] < 1e-10 and np.all(hist[n:] == 0)
        status, st = lq.lq_solve_MdagM(ctx, x, dev(phi), 0.14, 1e-11, 7, p, 30)
        assert status == lq.LQ_ERR_NOT_CONVERGED and st["iterations"] == 7
    finally:
        lq.lq_destroy(ctx)


def test_batch_with_a_context_replaced(lq):
    """The recorded solve graph of a batch holds its systems' links: a second context destroyed and
    created anew (at whatever addresses) between two solves is solved with its own links."""
    import torch
    dims, kappa = (4, 4, 4, 4), 0.15
    lat = Lattice(dims)
    phi = dev(source(lat, 3))
    first = lq.lq_create(dims)
    try:
        lq.lq_gauge_set(first, dev(gauge_exp_iA(lat, 0.3, 21)))
        for seed in (22, 23, 24):
            second = lq.lq_create(dims)
            try:
                lq.lq_gauge_set(second, dev(gauge_exp_iA(lat, 0.3, seed)))
                if seed == 23:              # other allocations in between
                    lq.lq_apply_M(second, torch.empty_like(phi), phi, kappa, False, lq.LQ_DF64)
                xs = [torch.zeros_like(phi), torch.zeros_like(phi)]
                status, st, _, resid, _ = lq.lq_solve_batch([first, second], xs, [phi, phi], [kappa, kappa], 1, 1e-10,
                                                            3000, lq.LQ_F16_12, 25)
                assert status == lq.LQ_OK and np.all(resid <= 1e-10)
                for c, x in zip((first, second), xs):
                    r = torch.empty_like(phi)
                    lq.lq_apply_MdagM(c, r, x, kappa, lq.LQ_F64)
                    assert float(torch.linalg.vector_norm(phi - r) / torch.linalg.vector_norm(phi)) <= 1.01e-10
            finally:
                lq.lq_destroy(second)
    finally:
        lq.lq_destroy(first)

"""Iterations replayed from a graph against the same launches from the host, on lattices beyond the cluster's."""
import numpy as np
import pytest

from synth import Lattice, gauge_exp_iA, source
from tests.gpu_common import require_gpu, dev, host, torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lq():
    return require_gpu()


@pytest.mark.parametrize("prec", ["f64", "f32", "f32_12", "f16_12", "bf16_12", "i16_12"])
def test_graphs_and_direct_launches_agree_to_the_bit(lq, prec):
    """The three kernels of an iteration overlap by programmatic launches, recorded in a graph or issued one by one:
    the same solution, history and counts.  6656 sites: more than run inside one cluster."""
    dims = (8, 8, 8, 13)
    lat = Lattice(dims)
    U, phi, p = dev(gauge_exp_iA(lat, 0.3, 8)), dev(source(lat, 8)), lq.PRECISIONS[prec]
    res = []
    for graphs in (1, 0):
        ctx = lq.lq_create(dims)
        try:
            lq.lq_set_option(ctx, lq.LQ_OPT_CUDA_GRAPHS, graphs)
            lq.lq_gauge_set(ctx, U)
            x, hist = torch.zeros_like(phi), np.zeros(3000)
            status, st = lq.lq_solve_MdagM(ctx, x, phi, 0.145, 1e-10, 3000, p, 40, hist=hist)
            assert status == lq.LQ_OK and st["true_rel_resid"] <= 1e-10
            res.append((host(x).copy(), hist, st["iterations"], st["reliable_updates"], st["kernel_launches"]))
        finally:
            lq.lq_destroy(ctx)
    assert np.array_equal(res[0][0], res[1][0]) and np.array_equal(res[0][1], res[1][1])
    assert res[0][2:] == res[1][2:]


@pytest.mark.parametrize("value", [0, 1])
def test_the_double_float_update_option_is_accepted_and_changes_nothing(lq, value):
    dims = (4, 4, 4, 4)
    lat = Lattice(dims)
    U, phi = dev(gauge_exp_iA(lat, 0.3, 8)), dev(source(lat, 8))
    out = []
    for option in (None, value):
        ctx = lq.lq_create(dims)
        try:
            if option is not None:
                lq.lq_set_option(ctx, lq.LQ_OPT_DF64_UPDATES, option)
            lq.lq_gauge_set(ctx, U)
            x = torch.zeros_like(phi)
            status, st = lq.lq_solve_MdagM(ctx, x, phi, 0.145, 1e-10, 3000, lq.LQ_F16_12, 25)
            assert status == lq.LQ_OK
            out.append((host(x).copy(), st["iterations"], st["kernel_launches"]))
        finally:
            lq.lq_destroy(ctx)
    assert np.array_equal(out[0][0], out[1][0])
    assert out[0][1] == out[1][1]

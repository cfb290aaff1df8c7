"""kernel_launches of a call against the kernels the profiler saw."""
import numpy as np
import pytest

from synth import Lattice, gauge_exp_iA, source
from tests.gpu_common import require_gpu, dev, torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lq():
    lib = require_gpu()
    from torch.profiler import ProfilerActivity, profile
    with profile(activities=[ProfilerActivity.CUDA]):       # its first window may come back empty
        torch.ones(8, device="cuda").sum().item()
    return lib


def _kernels(call):
    """Result of call() and how many kernels ran in it (copies and fills are not kernels)."""
    from torch.profiler import ProfilerActivity, profile
    torch.cuda.synchronize()
    with profile(activities=[ProfilerActivity.CUDA]) as prof:
        res = call()
        torch.cuda.synchronize()
    names = [e.name for e in prof.events() if e.device_type == torch.autograd.DeviceType.CUDA]
    if not names:
        pytest.skip("the profiler sees no kernels here")
    return res, sum(not n.lower().startswith(("memcpy", "memset")) for n in names)


@pytest.mark.parametrize("prec", ["f64", "f32_12"])
@pytest.mark.parametrize("dims", [(4, 4, 4, 4), (8, 8, 8, 14)])
def test_launches_of_solves_and_trajectories(lq, dims, prec):
    """Links freshly loaded, loaded before, and changed in every step of a trajectory."""
    lat = Lattice(dims)
    U, phi = dev(gauge_exp_iA(lat, 0.3, 5)), dev(source(lat, 5))
    x, p = torch.zeros_like(phi), lq.PRECISIONS[prec]
    ctx = lq.lq_create(dims)
    try:
        lq.lq_gauge_set(ctx, U)
        lq.lq_solve_MdagM(ctx, x, phi, 0.14, 1e-8, 2000, p, 20)         # graphs recorded, kernels loaded
        lq.lq_hmc_trajectory_seeded(ctx, 1, 0, 5.6, 0.14, 2, 0.1, 1e-8, 2000, p, 20)
        lq.lq_gauge_set(ctx, U)
        torch.cuda.synchronize()
        for _ in range(2):
            (status, st), n = _kernels(lambda: lq.lq_solve_MdagM(ctx, x, phi, 0.14, 1e-8, 2000, p, 20))
            assert status == lq.LQ_OK and st["kernel_launches"] == n
        res, n = _kernels(lambda: lq.lq_hmc_trajectory_seeded(ctx, 1, 1, 5.6, 0.14, 2, 0.1, 1e-8, 2000, p, 20))
        assert res["kernel_launches"] == n
    finally:
        lq.lq_destroy(ctx)
    assert np.isfinite(res["dH"])

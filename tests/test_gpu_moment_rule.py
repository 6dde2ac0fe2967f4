"""Which large FP32 boxes step on moments at tau = 1: those whose rows fill five eighths
of the warps of 32 that take them.  On either side of the line, and in boxes a cell
or two wide, the state and the read-outs are the staged kernel's.
"""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lbm():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1906_04722_gb300 as m
    m.load()
    with _profile():  # the first profile of a process may come back empty
        torch.zeros(1, device="cuda")
        torch.cuda.synchronize()
    return m


def _profile():
    from torch.profiler import ProfilerActivity, profile
    return profile(activities=[ProfilerActivity.CUDA])


@pytest.mark.parametrize("shape,moments", [
    ((820, 800, 1), False), ((600, 601, 2), False), ((216, 160, 19), False), ((200, 164, 20), True),
    ((130, 130, 39), False), ((130, 130, 40), True), ((97, 97, 97), True), ((1, 820, 832), True),
    ((600, 1, 1100), True), ((2, 600, 608), True),
])
def test_boxes_on_either_side(lbm, shape, moments):
    import torch
    import bench
    nz, ny, nx = shape
    p = lbm.make_params(periodic=(1, 1, 1))
    rho = W.droplet_densities(shape, (nx / 2, ny / 2, nz / 2), 0.25 * sorted(shape)[1], seed=5)
    got = []
    for kind in ("staged", "default"):
        d = lbm.Domain(p, None, (nx, ny, nz))
        d.set_densities(rho)
        if kind == "staged":
            d.set_step_kernel(lbm.KERNEL_STAGED)
        d.step(3)
        torch.cuda.synchronize()
        with _profile() as prof:
            d.step(2)
            torch.cuda.synchronize()
        names = {e.name for e in prof.events() if e.device_type == torch.autograd.DeviceType.CUDA}
        got.append((d.density(), d.state()[0], d.measure(), d.density_at(nx // 2, ny // 2, nz // 2)))
        d.close()
    a, b = got
    assert np.array_equal(a[0], b[0]) and np.array_equal(a[1], b[1]) and a[3] == b[3]
    assert a[2]["n_w"] == b[2]["n_w"] and a[2]["n_interface"] == b[2]["n_interface"]
    assert bench.on_moments((nx, ny, nz)) == moments
    if names:
        assert any("moment_gather_kernel" in n for n in names) == moments

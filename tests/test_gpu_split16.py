"""The two-launch step as a kernel of its own in 16-bit storage: LBM_KERNEL_SPLIT is
set, reported, timed and carried to another domain like any other kind, and
LBM_KERNEL_PUSH runs the push kernel whatever the size of the box.
"""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu

SPHERES = np.array([[9.0, 8.0, 7.0, 5.2], [24.0, 15.0, 19.0, 6.1], [30.5, 3.0, 26.0, 4.0]])


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


def _domain(lbm, shape, precision, spheres=SPHERES, **par):
    nz, ny, nx = shape
    p = lbm.make_params(G=W.G_COHESION, rho_major=W.RHO_MAJOR, rho_minor=W.RHO_MINOR, precision=precision, **par)
    d = lbm.Domain(p, spheres, (nx, ny, nz))
    d.set_densities(W.droplet_densities(shape, (nx / 2, ny / 2, nz / 2), 0.3 * min(shape) + 1, seed=5))
    return d


def _kernels(run):
    """Names of the kernels that run() launches."""
    import torch
    torch.cuda.synchronize()
    with _profile() as p:
        run()
        torch.cuda.synchronize()
    names = {e.name for e in p.events() if e.device_type == torch.autograd.DeviceType.CUDA}
    if not names:
        pytest.skip("the profiler records no kernels here")
    return names


@pytest.mark.parametrize("precision", [1, 2])
@pytest.mark.parametrize("shape,par", [((29, 21, 37), {}), ((53, 52, 52), {"reservoirs": True, "membrane_layers": 2}),
                                       ((31, 20, 34), {"periodic": (1, 1, 1)})])
def test_split_is_a_kind_of_its_own(lbm, precision, shape, par):
    staged = _domain(lbm, shape, precision, **par)
    staged.set_step_kernel(lbm.KERNEL_STAGED)
    staged.step(30)
    d = _domain(lbm, shape, precision, **par)
    d.set_step_kernel(lbm.KERNEL_SPLIT)
    assert d.step_kernel()[0] == lbm.KERNEL_SPLIT
    d.step(9)
    d.set_step_kernel(lbm.KERNEL_STAGED)
    d.step(4)
    d.set_step_kernel(lbm.KERNEL_SPLIT)
    names = _kernels(lambda: d.step(17))
    assert any("pair16_push_kernel" in n for n in names)
    assert np.array_equal(d.density(), staged.density())
    with pytest.raises(lbm.LbmError):
        _domain(lbm, shape, precision, tau=(0.8, 1.2), **par).set_step_kernel(lbm.KERNEL_SPLIT)


@pytest.mark.parametrize("shape", [(45, 29, 68), (54, 52, 52), (101, 102, 104)])
def test_push_is_the_push_kernel_at_every_size(lbm, shape):
    push, split = _domain(lbm, shape, 1), _domain(lbm, shape, 1)
    split.set_step_kernel(lbm.KERNEL_SPLIT)
    split.step(20)
    push.set_push_shape(3, 24)
    push.step(10)
    names = _kernels(lambda: push.step(10))
    assert any("sc_step16_push_kernel" in n for n in names) and not any("pair16" in n for n in names)
    assert np.array_equal(push.density(), split.density())


def test_sample192_push_and_split_agree(lbm):
    """The drainage sample in the shape that the sampled-cell check against the
    oracle uses for the push kernel."""
    shape, spheres = (192, 192, 192), W.sample192_spheres()
    got = []
    for kind in ("push", "split"):
        d = _domain(lbm, shape, 1, spheres, reservoirs=True, membrane_layers=3)
        if kind == "push":
            d.set_push_shape(3, 24)
        else:
            d.set_step_kernel(lbm.KERNEL_SPLIT)
        d.set_densities(W.initial_densities(shape, noise=2e-2, seed=8))
        d.step(2)
        got.append(d.density())
        d.close()
    assert np.array_equal(got[0], got[1])


@pytest.mark.parametrize("precision", [1, 2])
def test_a_tune_result_carries_over(lbm, precision):
    """On a box that the push kernel does not serve, the two-launch step is the
    fastest by far: the result names it, and takes a second domain to it."""
    shape = (62, 60, 61)
    a = _domain(lbm, shape, precision)
    res = a.autotune(trial_steps=20)
    assert res["kind"] == "split" and a.step_kernel()[0] == lbm.KERNEL_SPLIT
    b = _domain(lbm, shape, precision)
    b.set_step_kernel(lbm.KERNEL_SPLIT)
    a.step(8)
    b.step(8)
    assert _kernels(lambda: a.step(3)) == _kernels(lambda: b.step(3))
    assert np.array_equal(a.density(), b.density())

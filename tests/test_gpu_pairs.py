"""The two-launch step (LBM_KERNEL_SPLIT, and the route of a domain without a
chosen kernel) against the staged kernel, bit for bit: ragged and odd boxes, every
periodic axis, boxes one or two cells wide, membrane and reservoirs, body force,
boxes large enough to step on moments; switching kernels on the way; at tau = 1 and
at others.
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
    return m


def _domain(lbm, shape, periodic, **par):
    nz, ny, nx = shape
    p = lbm.make_params(rho_major=W.RHO_MAJOR, rho_minor=W.RHO_MINOR, periodic=periodic, **par)
    d = lbm.Domain(p, SPHERES, (nx, ny, nz))
    d.set_densities(W.droplet_densities(shape, (nx / 2, ny / 2, nz / 2), 0.3 * min(shape) + 1, seed=5))
    return d


def _read(d, steps):
    d.step(steps)
    f, st = d.state()
    return f, st, d.density(), d.measure(allow_nonfinite=True)


def _equal(a, b):
    assert np.array_equal(a[0], b[0]) and a[1] == b[1] and np.array_equal(a[2], b[2])
    for k in ("n_fluid", "n_w", "n_interface", "n_bulk_w", "n_bulk_nw", "n_in", "n_out", "n_negative"):
        assert a[3][k] == b[3][k]
    assert np.allclose(a[3]["mass"], b[3]["mass"], rtol=1e-12, atol=0)


@pytest.mark.parametrize("shape,periodic,par", [
    ((29, 21, 37), (0, 0, 0), {}),
    ((30, 23, 33), (1, 0, 0), {}),
    ((31, 20, 34), (0, 1, 1), {"body_force": (1e-5, -2e-5, 3e-5)}),
    ((16, 17, 18), (1, 1, 1), {"G_ads": (0.0, 0.0)}),
    ((40, 22, 35), (0, 0, 0), {"reservoirs": True, "membrane_layers": 3}),
    ((9, 1, 40), (0, 1, 0), {}),
    ((2, 19, 2), (1, 1, 1), {}),
    ((90, 87, 89), (0, 0, 0), {"reservoirs": True, "membrane_layers": 3}),
    ((91, 88, 87), (1, 1, 1), {"body_force": (1e-5, -2e-5, 3e-5)}),
])
def test_equals_the_staged_kernel(lbm, shape, periodic, par):
    staged = _domain(lbm, shape, periodic, **par)
    staged.set_step_kernel(lbm.KERNEL_STAGED)
    want = _read(staged, 70)
    default = _domain(lbm, shape, periodic, **par)
    assert default.step_kernel()[0] == lbm.KERNEL_STAGED
    _equal(_read(default, 70), want)
    split = _domain(lbm, shape, periodic, **par)
    split.step(13)
    split.set_step_kernel(lbm.KERNEL_SPLIT)
    split.step(30)
    split.set_step_kernel(lbm.KERNEL_STAGED)
    split.step(8)
    split.set_step_kernel(lbm.KERNEL_SPLIT)
    _equal(_read(split, 19), want)
    # a checkpoint into another domain, densities reset, and the staged kernel after
    # another layout was in its buffers: grain cells keep their zeros
    f, st = split.state()
    other = _domain(lbm, shape, periodic, **par)
    other.step(3)
    other.set_state(f, st)
    other.step(2)
    staged.step(2)
    _equal(_read(other, 1), _read(staged, 1))
    other.set_step_kernel(lbm.KERNEL_STAGED)
    _equal(_read(other, 3), _read(staged, 3))
    for d in (other, staged):
        d.set_densities(W.droplet_densities(shape, (1, 2, 3), 4.0, seed=6))
    _equal(_read(other, 5), _read(staged, 5))
    nx, ny, nz = other.dims
    assert other.density_at(nx // 2, ny // 2, nz // 2) == staged.density_at(nx // 2, ny // 2, nz // 2)


def test_unequal_tau(lbm):
    a = _domain(lbm, (21, 18, 27), (0, 0, 1), tau=(1.0, 1.2))
    b = _domain(lbm, (21, 18, 27), (0, 0, 1), tau=(1.0, 1.2))
    b.set_step_kernel(lbm.KERNEL_STAGED)
    _equal(_read(a, 20), _read(b, 20))
    c = _domain(lbm, (21, 18, 27), (0, 0, 1), tau=(1.0, 1.2))
    c.set_step_kernel(lbm.KERNEL_SPLIT)
    c.step(20)
    assert np.allclose(c.density(), a.density(), rtol=1e-5, atol=1e-7)


@pytest.mark.parametrize("tau", [(0.8, 1.2), (1.0, 1.2), (0.7, 0.7)])
@pytest.mark.parametrize("shape,periodic,par", [
    ((29, 21, 37), (0, 0, 0), {}),
    ((31, 20, 34), (0, 1, 1), {"body_force": (1e-5, -2e-5, 3e-5)}),
    ((40, 22, 35), (0, 0, 0), {"reservoirs": True, "membrane_layers": 3}),
    ((9, 1, 40), (0, 1, 0), {}),
    ((2, 19, 2), (1, 1, 1), {}),
    ((90, 87, 89), (0, 0, 1), {}),
])
def test_any_tau_equals_the_staged_kernel(lbm, shape, periodic, par, tau):
    staged = _domain(lbm, shape, periodic, tau=tau, **par)
    staged.set_step_kernel(lbm.KERNEL_STAGED)
    want = _read(staged, 70)
    _equal(_read(_domain(lbm, shape, periodic, tau=tau, **par), 70), want)
    d = _domain(lbm, shape, periodic, tau=tau, **par)
    d.step(13)
    d.set_step_kernel(lbm.KERNEL_STAGED)
    d.step(30)
    d.set_step_kernel(lbm.KERNEL_SPLIT)
    _equal(_read(d, 27), want)


@pytest.mark.parametrize("precision", [1, 2])
@pytest.mark.parametrize("shape,periodic,par", [
    ((29, 21, 37), (0, 0, 0), {}),
    ((31, 20, 34), (1, 1, 1), {"body_force": (1e-5, -2e-5, 3e-5)}),
    ((40, 22, 35), (0, 0, 0), {"reservoirs": True, "membrane_layers": 3}),
    ((2, 19, 2), (1, 1, 1), {}),
    ((52, 51, 52), (0, 0, 1), {}),
    ((101, 102, 104), (0, 0, 0), {"reservoirs": True, "membrane_layers": 2}),
])
def test_16_bit(lbm, precision, shape, periodic, par):
    """Untuned, and (from 2^17 cells on) as the push kernel; the last box is one
    of 2^20 cells and more, whose second launch reads the densities twice."""
    staged = _domain(lbm, shape, periodic, precision=precision, **par)
    staged.set_step_kernel(lbm.KERNEL_STAGED)
    default = _domain(lbm, shape, periodic, precision=precision, **par)
    push = _domain(lbm, shape, periodic, precision=precision, **par)
    for d in (staged, default):
        d.step(31)
    if shape[2] % 4 == 0 and not periodic[0]:
        push.step(9)
        push.set_step_kernel(lbm.KERNEL_PUSH)
        push.step(11)
        push.set_step_kernel(lbm.KERNEL_STAGED)
        push.step(5)
        push.set_push_shape(0, 8)
        push.step(6)
    else:
        push.step(31)
    for d in (default, push):
        assert np.array_equal(d.density(), staged.density())
        a, b = d.measure(allow_nonfinite=True), staged.measure(allow_nonfinite=True)
        assert a["n_w"] == b["n_w"] and a["n_interface"] == b["n_interface"]
        assert d.density_at(1, 5, 1) == staged.density_at(1, 5, 1)


@pytest.mark.parametrize("precision,par,shape", [
    (0, {}, (29, 21, 37)), (1, {}, (29, 21, 37)), (0, {"tau": (0.8, 1.2)}, (29, 21, 37)), (0, {}, (90, 87, 89)),
])
def test_short_runs_equal_one_long_run(lbm, precision, par, shape):
    runs = [7, 8, 25, 9, 31, 8, 63, 25]  # chunks of 8 replay a graph from the fourth run of 8 and more on
    a = _domain(lbm, shape, (0, 0, 1), precision=precision, **par)
    b = _domain(lbm, shape, (0, 0, 1), precision=precision, **par)
    b.set_step_kernel(lbm.KERNEL_STAGED)
    b.step(sum(runs) + 2 * 20)
    for n in runs:
        a.step(n)
    a.set_step_kernel(lbm.KERNEL_STAGED)  # drops the graphs
    a.step(20)
    a.step(20)
    if precision == 0:
        _equal(_read(a, 0), _read(b, 0))
    assert np.array_equal(a.density(), b.density())

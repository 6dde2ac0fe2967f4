"""What a failing call leaves behind.  The failure is the host's: while a stream of the
process is captured in global mode, the runtime refuses the calls that wait.
"""
import contextlib
import ctypes
import threading
import time

import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu

SPHERES = np.array([[20.0, 18.0, 17.0, 11.2], [64.0, 55.0, 49.0, 16.1], [70.5, 13.0, 66.0, 14.0]])
SHAPE = (92, 90, 88)


@pytest.fixture(scope="module")
def lbm():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1906_04722_gb300 as m
    m.load()
    return m


@contextlib.contextmanager
def _waits_refused():
    import torch
    torch.cuda.synchronize()
    rt = ctypes.CDLL("libcudart.so.%s" % torch.version.cuda.split(".")[0])
    stream, graph = ctypes.c_void_p(), ctypes.c_void_p()
    assert rt.cudaStreamCreateWithFlags(ctypes.byref(stream), 1) == 0
    assert rt.cudaStreamBeginCapture(stream, 0) == 0
    try:
        yield
    finally:
        if rt.cudaStreamEndCapture(stream, ctypes.byref(graph)) == 0 and graph:
            rt.cudaGraphDestroy(graph)
        rt.cudaStreamDestroy(stream)
        rt.cudaGetLastError()


def _in_thread(call):
    """Runs call() in a thread of its own (the runtime keeps its last error by thread)."""
    got = []

    def work():
        try:
            got.append(call())
        except Exception as e:  # handed to the caller
            got.append(e)
    t = threading.Thread(target=work)
    t.start()
    return t, got


def _domain(lbm, precision=0):
    import torch
    nz, ny, nx = SHAPE
    p = lbm.make_params(rho_major=W.RHO_MAJOR, rho_minor=W.RHO_MINOR, precision=precision)
    d = lbm.Domain(p, SPHERES, (nx, ny, nz), stream=torch.cuda.Stream().cuda_stream)
    d.set_densities(W.droplet_densities(SHAPE, (nx / 2, ny / 2, nz / 2), 20.0, seed=5))
    return d


def test_a_failed_autotune_leaves_the_domain_as_it_was(lbm):
    """In the pull layout grain cells hold zeros in both buffers, whatever layout the
    candidates timed so far stepped on."""
    d, ref = _domain(lbm), _domain(lbm)
    for x in (d, ref):
        x.set_tile(8, 16, 2)
        x.step(2)
    t, got = _in_thread(lambda: d.autotune(trial_steps=60))
    time.sleep(0.3)
    with _waits_refused():
        t.join()
    if not isinstance(got[0], lbm.LbmError):
        pytest.skip("the tuning was over before it could fail")
    assert d.tile() == (8, 16, 2)
    for n in (1, 2):
        d.step(n)
        ref.step(n)
        a, b = d.state(), ref.state()
        assert np.array_equal(a[0], b[0]) and a[1] == b[1]


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("call", ["density", "state"])
def test_a_failed_read_out_leaves_the_array_as_it_was(lbm, call, precision):
    if call == "state" and precision:
        pytest.skip("16-bit domains have no checkpoints")
    d = _domain(lbm, precision)
    d.step(3)
    n = int(np.prod(SHAPE)) * (2 if call == "density" else 38)
    out = np.full(n, 7.0, np.float64 if call == "density" else np.float32)
    L = lbm.load()
    if call == "density":
        def read():
            return L.lbm_get_density(d.h, out.ctypes.data_as(ctypes.POINTER(ctypes.c_double)))
    else:
        step = ctypes.c_longlong(0)

        def read():
            return L.lbm_get_state(d.h, out.ctypes.data_as(ctypes.POINTER(ctypes.c_float)), ctypes.byref(step))
    with _waits_refused():
        t, got = _in_thread(read)
        t.join()
    assert got[0] != 0
    assert np.all(out == 7.0)
    assert read() == 0
    want = d.density() if call == "density" else d.state()[0]
    assert np.array_equal(out, want.ravel())


@pytest.mark.parametrize("precision", [0, 2])
@pytest.mark.parametrize("shape", [(1, 1, 1), (16, 32, 32), (17, 32, 32)])
def test_densities_converted_by_the_host_or_the_device(lbm, shape, precision):
    """2^15 values are the largest field that the host converts."""
    nz, ny, nx = shape
    d = lbm.Domain(lbm.make_params(periodic=(1, 1, 1), precision=precision), None, (nx, ny, nz))
    rho = W.droplet_densities(shape, (nx / 2, ny / 2, nz / 2), 6.0, seed=5)
    d.set_densities(rho)
    got = d.density()
    want = rho.astype(np.float32)
    assert np.allclose(got, want, rtol=1e-6, atol=0)  # the sum of 19 rest populations
    assert np.array_equal(got, got.astype(np.float32))
    for z, y, x in ((0, 0, 0), (nz - 1, ny - 1, nx - 1), (nz // 2, ny // 3, nx // 4)):
        assert tuple(got[:, z, y, x]) == tuple(d.density_at(x, y, z))

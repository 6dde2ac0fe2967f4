"""Steps that a caller captures in a CUDA graph of its own and replays, on domains of
the two-launch route: the state is the staged kernel's after as many steps, whether
the domain was stepped before the capture or not, mixed with steps of the library's
own, and after the state has been set anew.
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


@pytest.mark.parametrize("warm", [0, 2, 5, 40])
@pytest.mark.parametrize("kind", ["unchosen", "split"])
@pytest.mark.parametrize("shape,par", [
    ((29, 21, 37), {}),
    ((29, 21, 37), {"tau": (0.8, 1.2)}),
    ((30, 22, 35), {"reservoirs": True, "membrane_layers": 3, "precision": 1}),
    ((29, 21, 37), {"precision": 2, "periodic": (1, 0, 1)}),
    ((90, 87, 89), {}),
])
def test_captured_steps_replay(lbm, shape, par, kind, warm):
    import torch
    nz, ny, nx = shape
    p = lbm.make_params(rho_major=W.RHO_MAJOR, rho_minor=W.RHO_MINOR, **par)
    rho = [W.droplet_densities(shape, (nx / 2, ny / 2, nz / 2), 0.3 * min(shape) + 1, seed=s) for s in (5, 6)]
    s = torch.cuda.Stream()
    d = lbm.Domain(p, SPHERES, (nx, ny, nz), stream=s.cuda_stream)
    ref = lbm.Domain(p, SPHERES, (nx, ny, nz))
    ref.set_step_kernel(lbm.KERNEL_STAGED)
    for x in (d, ref):
        x.set_densities(rho[0])
    if kind == "split":
        d.set_step_kernel(lbm.KERNEL_SPLIT)

    def same():
        assert np.array_equal(d.density(), ref.density())
        if par.get("precision", 0) == 0:
            assert np.array_equal(d.state()[0], ref.state()[0])

    d.step(warm)
    ref.step(warm)
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=s):
        d.step(4)
    same()  # a capture runs nothing

    def replay(n):
        with torch.cuda.stream(s):
            for _ in range(n):
                g.replay()
        ref.step(4 * n)
        same()

    replay(3)
    d.step(66)
    ref.step(66)
    replay(1)
    for x in (d, ref):
        x.set_densities(rho[1])
    replay(2)
    if par.get("precision", 0) == 0:
        f, st = ref.state()
        d.set_state(f, st)
        replay(1)

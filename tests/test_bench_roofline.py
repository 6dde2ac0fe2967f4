"""The bytes that bench.py charges a step, and the sources behind its traffic records."""
import os
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
sys.path.insert(0, ROOT)
import bench  # noqa: E402


@pytest.mark.parametrize("name,per_cell,source", [
    ("moment_gather_kernel + moment_collide_kernel (one step)", 136, "lbm_step_moments.cu"),
    ("pair_moment_kernel + pair_push_kernel (one step)", 344, "lbm_step_pairs.cu"),
    ("pair_moment_kernel + pair_relax_kernel (one step)", 472, "lbm_step_pairs.cu"),
    ("pair16_moment_kernel<half2> + pair16_push_kernel<half2> (one step)", 200, "lbm_step16_pairs.cu"),
])
def test_two_launch_steps(name, per_cell, source):
    """What the route moves, not the populations that it may not even keep."""
    got, bound = bench.step_bytes(name, 1000, 304000)
    assert got == 1000 * per_cell
    assert bound != "hbm" or "relax" in name
    key = next(k for k in bench.KERNEL_SOURCES if name.startswith(k))
    assert bench.KERNEL_SOURCES[key][0] == source
    assert bench.kernel_hash(name) != bench.kernel_hash("sc_step_kernel<6,2>")


@pytest.mark.parametrize("name", ["sc_step_push_kernel<6,3,2,true,true>", "sc_step_kernel<6,2>", "sc_step_tma_kernel",
                                  "sc_step16_push_kernel<half2,10,3,2>"])
def test_one_launch_steps(name):
    assert bench.step_bytes(name, 1000, 304000) == (304000, "hbm")
    for f in bench.KERNEL_SOURCES[next(k for k in bench.KERNEL_SOURCES if name.startswith(k))]:
        assert os.path.exists(os.path.join(ROOT, "paper_1906_04722_gb300", "csrc", f))

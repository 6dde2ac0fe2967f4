"""The throat batch's on-chip form (AUTO at tau = 1) against the cell list.

Both run the same arithmetic in the same order, so the rows must agree bit for
bit: throats from a few hundred cells (one CTA) to the largest a cluster holds
and beyond (those stay with the cell list beside it), one and two cells per
thread, ranges that end inside a plane, odd and even step counts, none at all,
one ladder for all or one each, a body force.
"""
import math

import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu

KEYS = ("rho_in_nw", "p_c", "p_c_res", "S_w", "p_w", "p_nw", "phi_probe", "n_interface")


@pytest.fixture(scope="module")
def lbm():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1906_04722_gb300 as m
    m.load()
    return m


def _throat(r, gap):
    """Three spheres of radius r on an equilateral triangle, gap between the surfaces."""
    side = 2.0 * r + gap
    R = side / math.sqrt(3.0)
    return [(R * math.cos(a) + 0.3, R * math.sin(a) - 0.2, 0.1, r) for a in (0.4, 0.4 + 2 * math.pi / 3, 0.4 + 4 * math.pi / 3)]


def _same(lbm, throats, params, ladder, steps):
    th = np.asarray(throats, dtype=float)
    (ra, wa), (rb, wb) = (lbm.lbm_run_throat_batch(th, params, ladder, steps, W.RHO_MAJOR, form=f)
                          for f in (lbm.BATCH_AUTO, lbm.BATCH_CELLS))
    for f in ("invaded_at", "dims", "probe", "n_fluid", "p_ce"):
        assert [r[f] for r in ra] == [r[f] for r in rb]
    a, b = (np.array([[[r[k] for k in KEYS] for r in t] for t in w]) for w in (wa, wb))
    assert np.array_equal(a, b, equal_nan=True)
    return [r["n_fluid"] for r in ra]


# (radius, gap): about 250 to 40 000 open cells
SIZES = [(5.0, 0.5), (7.0, 2.0), (10.0, 0.0), (11.0, 6.0), (13.0, 9.0), (14.0, 14.0), (16.0, 20.0), (17.0, 26.0)]


@pytest.mark.parametrize("steps", [0, 1, 26, 33])
def test_sizes_one_by_one(lbm, steps):
    p = lbm.make_params(body_force=(1e-5, -2e-5, 3e-5))
    cells = [_same(lbm, [_throat(r, g)], p, [2.0, 2.08], steps)[0] for r, g in SIZES]
    assert min(cells) < 1024 and max(cells) > 16 * 1408  # one CTA; more than a cluster holds


@pytest.mark.parametrize("n", [2, 17, 60])
def test_mixed_batches(lbm, n):
    rng = np.random.default_rng(n)
    throats = [_throat(rng.uniform(5, 17), rng.uniform(0, 22)) for _ in range(n)]
    ladders = 2.0 + rng.uniform(0, 0.1, (n, 3))
    _same(lbm, throats, lbm.make_params(), ladders, 25)


def test_other_tau_stays_with_the_cell_list(lbm):
    _same(lbm, [_throat(8.0, 3.0), _throat(12.0, 8.0)], lbm.make_params(tau=(1.0, 1.1)), [2.0, 2.05], 20)

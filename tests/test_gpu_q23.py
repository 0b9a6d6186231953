"""The Q2 3D FP32 sweep (a warp copies the rows of 32 due elements together) at the edges of its
tiles -- one element, a partial warp, a warp and one, several blocks -- for the pointwise forms it
has, against the FP64 oracle.

Tolerance: 4 barrier steps of at most 4 substeps, each rounding V and v to FP32 (6e-8 relative)
and the increment's terms to a few 6e-8 of the local variation: 16 x 6e-8 x 4 = 4e-6, held to 1e-5.
"""
import numpy as np
import pytest

import workloads as W
from oracle import lts
from tests.helpers import mass_rel_l2

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def mdl():
    import torch
    if not torch.cuda.is_available():
        pytest.fail("CUDA device required for -m gpu tests")
    from paper_2310_07607_gb300 import build, mdl as M
    build.build()
    return M


@pytest.mark.parametrize("base,form", [((1, 1, 1), "exp"), ((31, 1, 1), "exp"), ((32, 1, 1), "fe"), ((33, 1, 1), "exp"),
                                       ((43, 3, 1), "none"), ((13, 5, 2), "stim2"), ((11, 4, 3), "oblique")])
def test_q23_tile_edges(mdl, base, form):
    prob = W.scaled(W.slab_3d_q2(), base).replace(amr_enabled=0, max_refine=0, n_lts_levels=3)
    if form == "fe":
        prob = prob.replace(state_integrator=W.STATE_FE)
    if form == "none":
        prob = prob.replace(ionic_model=-1, stimuli=[])
    if form == "stim2":
        e = prob.extent
        prob = prob.replace(stimuli=[W.Stimulus((0, 0, 0), (0.4 * e[0], e[1], e[2]), 0.7, 0.0, 1.0),
                                     W.Stimulus((0.2 * e[0], 0, 0), (e[0], 0.5 * e[1], e[2]), 0.4, 0.0, 1e-3)])
    if form == "oblique":
        prob = prob.replace(fibre=(0.48, 0.64, 0.6))
    o = lts.Sim(prob)
    V0, v0 = W.planar_front_state(o.disc.node_coords(), 0.45 * prob.extent[0], 0.012, 0.3)
    o.V, o.v = V0.copy(), v0.copy()
    g = mdl.Sim(prob)
    g.set_sweep_variant(mdl.SWEEP_THREAD)
    g.set_initial(V0, v0)
    for _ in range(4):
        o.barrier()
    g.step_barriers(4)
    assert mass_rel_l2(o.disc.M, g.read_V(), o.V) <= 1e-5
    assert np.abs(g.read_state() - o.v).max() <= 1e-5 * max(np.abs(o.v).max(), 1.0)
    assert np.allclose(g.read_indicators()[1], o.eta_t, rtol=1e-2, atol=1e-4 * max(o.eta_t.max(), 1e-300))
    g.close()

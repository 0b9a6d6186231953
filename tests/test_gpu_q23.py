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
from tests.helpers import forest_arrays, mass_rel_l2, random_forest

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


@pytest.mark.parametrize("fibre", [(1.0, 0.0, 0.0), (0.48, 0.64, 0.6)])
@pytest.mark.parametrize("seed", [2, 4])
def test_q23_graded_mesh_and_indicator(mdl, fibre, seed):
    """Coarser and finer faces, which load in their own path, within the warps' row copies; a last warp
    of every tick that is not full; and the indicator kernel with the same copies.  Indicator: a flux
    jump is a sum of a few differences of shifted values of at most 1, each rounded to 6e-8, times
    derivative weights of at most 6: 4e-6 of the front's jumps (0.1 and more), held to 1e-4 of the
    largest."""
    prob = W.Problem(dim=3, order=2, extent=(0.4, 0.3, 0.2), base=(4, 3, 2), sigma_l=1.2, sigma_t=0.4, fibre=fibre,
                     gamma=40.0, max_refine=2, n_lts_levels=3, lts_enabled=1, amr_enabled=1, tau_refine=1e30,
                     tau_coarsen=-1.0, dt_barrier=0.0, state_integrator=W.STATE_EXP, precision=32,
                     stimuli=[W.Stimulus((0, 0, 0), (0.1, 0.1, 0.1), 1.0, 0.0, 1.0)])
    f = random_forest(3, prob.base, 2, prob.extent, steps=2, seed=seed, tau=0.7)
    o = lts.Sim(prob, forest=f)
    V0, v0 = W.front_state(o.disc.node_coords(), (0, 0, 0), 0.15, 0.02, tail=0.05)
    V0, v0 = V0.astype(np.float32).astype(np.float64), v0.astype(np.float32).astype(np.float64)
    o.V, o.v = V0.copy(), v0.copy()
    g = mdl.Sim(prob)
    g.upload_mesh(*forest_arrays(f))
    g.set_initial(V0, v0)
    g.step_barriers(1)
    want = o.disc.eta_s(V0)
    assert np.abs(g.read_indicators()[0] - want).max() <= 1e-4 * want.max()
    g.step_barriers(3)
    due = []
    for _ in range(4):
        lev = o.assign_levels(o.eta_t)
        due += [int((lev >= b).sum()) for b in range(lev.max() + 1)]
        o.eta_t = o.sweep(lev)
        o.barrier_count += 1
    assert any(n % 32 for n in due) and lev.max() > lev.min()
    assert mass_rel_l2(o.disc.M, g.read_V(), o.V) <= 1e-5
    assert np.abs(g.read_state() - o.v).max() <= 1e-5 * max(np.abs(o.v).max(), 1.0)
    g.close()


def test_q23_warps_that_walk_many_elements(mdl):
    """One block of 64 threads per SM: a warp takes a second, third and later group of 32 due elements of
    an adapting mesh, whose metadata it fetched a step ahead.  The same bits as with a warp a group."""
    prob = W.scaled(W.slab_3d_q2(), (30, 13, 5))
    a, b = mdl.Sim(prob), mdl.Sim(prob)
    b.set_tick_shape(64, 1)
    x = np.arange(prob.n_base) % prob.base[0]
    V = np.repeat(0.5 * (1.0 - np.tanh((x - 14.0) / 1.5)), 27)
    for g in (a, b):
        g.set_initial(V, np.zeros_like(V))
        g.step_barriers(6)
    assert a.sizes()[0] > 3 * 64 * 152
    for p, q in zip(a.read_mesh(), b.read_mesh()):
        assert np.array_equal(p, q)
    assert np.array_equal(a.read_V(), b.read_V()) and np.array_equal(a.read_state(), b.read_state())
    a.close()
    b.close()

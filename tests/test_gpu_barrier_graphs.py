"""Barriers replayed several to a graph, and the lane-per-DOF sweep that small Q1 meshes take when no
variant is asked for.

A run in one call (graphs of four barriers after the first 48) must give the bits of the same run one
barrier per call: the kernels and their order are the same.  The two Q1 sweeps sum the same terms in
another order: 60 barriers of at most 4 substeps, each within a few roundings of the local terms --
240 x 6e-8 = 1.4e-5 in FP32 (held to 2e-5 of the largest value), 240 x 1.1e-16 in FP64 (held to 1e-12).
"""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def mdl():
    import torch
    if not torch.cuda.is_available():
        pytest.fail("CUDA device required for -m gpu tests")
    from paper_2310_07607_gb300 import build, mdl as M
    build.build()
    return M


def problem(dim, order, precision, amr):
    base = (13, 9, 1) if dim == 2 else (7, 4, 3)
    h = (8.0 * 0.0078125 if dim == 2 else 4.0 * 0.015625) * order
    ext = tuple(base[k] * h if k < dim else 1.0 for k in range(3))
    tau = W.COMPLETED_TAU[(dim, order)]
    return W.Problem(dim=dim, order=order, extent=ext, base=base, sigma_l=1.2, sigma_t=0.4,
                     fibre=W.fibre_from_angle(0.6), gamma=10.0 * order * order,
                     stimuli=[W.Stimulus((0.0, 0.0, 0.0), tuple(0.2 * e for e in ext), 1.0, 0.0, 1.0)],
                     dt_barrier=0.0, max_refine=2 if amr else 0, n_lts_levels=3, tau_cell=0.5, tau_refine=tau[0],
                     tau_coarsen=tau[1], state_integrator=W.STATE_EXP, precision=precision, amr_enabled=amr,
                     lts_enabled=1)


@pytest.mark.parametrize("dim,order,precision,amr", [(2, 1, 32, 1), (2, 2, 32, 1), (3, 1, 64, 1), (3, 2, 32, 1),
                                                     (2, 1, 64, 0), (3, 2, 32, 0)])
def test_series_of_barriers_give_the_bits_of_single_steps(mdl, dim, order, precision, amr):
    p = problem(dim, order, precision, amr)
    n = 119                                     # 48 one by one, 17 series of four, 3 more
    a, b = mdl.Sim(p), mdl.Sim(p)
    for _ in range(n):
        a.step_barriers(1)
    b.step_barriers(n)
    assert a.time()[1] == b.time()[1] == n
    for x, y in zip(a.read_mesh(), b.read_mesh()):
        assert np.array_equal(x, y)
    assert np.array_equal(a.read_V(), b.read_V()) and np.array_equal(a.read_state(), b.read_state())
    assert np.array_equal(a.read_activation(), b.read_activation())
    for k in ("dof_updates", "tick_launches", "kernel_launches", "amr_rebuilds", "integral_V"):
        assert a.stats()[k] == b.stats()[k], k
    a.close()
    b.close()


@pytest.mark.parametrize("dim,precision,amr", [(2, 32, 0), (2, 64, 0), (3, 32, 0), (2, 64, 1), (3, 64, 1)])
def test_small_q1_default_sweep_matches_the_thread_sweep(mdl, dim, precision, amr):
    p = problem(dim, 1, precision, amr)
    a, b = mdl.Sim(p), mdl.Sim(p)
    b.set_sweep_variant(mdl.SWEEP_THREAD)
    a.step_barriers(60)
    b.step_barriers(60)
    assert np.array_equal(a.read_mesh()[1], b.read_mesh()[1])
    tol = 2e-5 if precision == 32 else 1e-12
    for x, y in ((a.read_V(), b.read_V()), (a.read_state(), b.read_state())):
        assert np.abs(x - y).max() <= tol * max(np.abs(y).max(), 1e-30)
    a.close()
    b.close()


@pytest.mark.parametrize("precision", [32, 64])
def test_an_uploaded_mesh_runs_as_in_a_new_context(mdl, precision):
    """900 root elements, then 3600 uploaded within the capacity, then 900 again: launch shapes and the
    choice of the sweep follow the mesh that is stepped, not the one that was stepped before it."""
    p = problem(2, 1, precision, 0).replace(base=(30, 30, 1), extent=(1.9, 1.9, 1.0), max_refine=1, stimuli=[],
                                            dt_barrier=2.0 ** -8)

    def mesh(level):
        n = 30 << level
        block = 1 << level                       # leaves in root order, then Morton order
        xy = [(i * block + a, j * block + b) for j in range(30) for i in range(30)
              for b in range(block) for a in range(block)]
        assert len(xy) == n * n
        return np.full(n * n, level, np.int8), np.array(xy, np.int32)

    used = mdl.Sim(p)
    for level in (0, 1, 0):
        V = 0.5 + 0.5 * np.sin(np.arange((900 << (2 * level)) * 4) / 91.0)
        new = mdl.Sim(p)
        for g in (used, new):
            g.upload_mesh(*mesh(level))
            g.set_initial(V, 0.3 * V)
            g.step_barriers(60)
        assert np.array_equal(used.read_V(), new.read_V()) and np.array_equal(used.read_state(), new.read_state())
        assert np.array_equal(used.read_indicators()[1], new.read_indicators()[1])
        new.close()
    used.close()


# roots (adapting) or elements (fixed) at both sides of the line between the two Q1 sweeps: DOFs per SM
@pytest.mark.parametrize("dim,precision,amr,depth,dofs_per_sm", [(2, 64, 0, 0, 128), (3, 64, 0, 0, 128), (2, 64, 1, 2, 128),
                                                                (2, 32, 1, 2, 108), (3, 32, 1, 2, 108), (2, 32, 1, 3, 54),
                                                                (2, 32, 0, 0, 0), (3, 32, 0, 0, 0)])
def test_default_q1_sweep_is_the_one_stated(mdl, dim, precision, amr, depth, dofs_per_sm):
    import torch
    nsm = torch.cuda.get_device_properties(0).multi_processor_count
    last = nsm * dofs_per_sm // 2 ** dim          # most elements that take a lane per DOF
    for n, variant in ((last, mdl.SWEEP_GROUP), (last + 1, mdl.SWEEP_THREAD)):
        if n == 0:
            continue
        rows = max(k for k in range(1, 41) if n % k == 0)
        base = (n // rows, rows, 1)
        p = problem(dim, 1, precision, amr).replace(base=base, extent=(0.06 * base[0], 0.06 * base[1], 0.06),
                                                    max_refine=depth, dt_barrier=0.0)
        V = 0.5 + 0.5 * np.sin(np.arange(n * 2 ** dim) / 91.0)
        a, b = mdl.Sim(p), mdl.Sim(p)
        b.set_sweep_variant(variant)
        for g in (a, b):
            g.set_initial(V, 0.3 * V)
            g.step_barriers(12)
        assert np.array_equal(a.read_mesh()[1], b.read_mesh()[1])
        assert np.array_equal(a.read_V(), b.read_V()) and np.array_equal(a.read_state(), b.read_state())
        a.close()
        b.close()


@pytest.mark.parametrize("dim,precision", [(2, 32), (3, 32), (2, 64)])
def test_adapting_run_does_not_depend_on_the_capacity(mdl, dim, precision):
    """A context whose capacity grows during the run against one that had room from the start."""
    base = (32, 32, 1) if dim == 2 else (16, 12, 8)
    p = problem(dim, 1, precision, 1).replace(base=base, extent=tuple(b / 64.0 for b in base), max_refine=3, tau_refine=1e-12,
                                              tau_coarsen=1e-13, dt_barrier=0.0, stimuli=[])
    xy = [(i, j, k)[:dim] for k in range(base[2]) for j in range(base[1]) for i in range(base[0])]
    roots = (np.zeros(len(xy), np.int8), np.array(xy, np.int32))
    n1 = 2 ** dim                                   # every root's children, in Morton order
    kids = (np.ones(len(xy) * n1, np.int8),
            np.array([[2 * c[t] + ((b >> t) & 1) for t in range(dim)] for c in xy for b in range(n1)], np.int32))
    small, large = mdl.Sim(p), mdl.Sim(p)
    if dim == 2:                                    # level 2: 16384 leaves, capacity 32768
        kids = (np.full(len(xy) * 16, 2, np.int8), np.array(
            [(4 * i + (b & 1) + 2 * ((b >> 2) & 1), 4 * j + ((b >> 1) & 1) + 2 * ((b >> 3) & 1)) for i, j in xy
             for b in range(16)], np.int32))
    large.upload_mesh(*kids)
    large.upload_mesh(*roots)
    x = np.repeat(np.array(xy)[:, 0], 2 ** dim).astype(float)
    V = 0.5 * (1.0 - np.tanh((x - 0.5 * base[0]) / 2.0))
    for g in (small, large):
        g.set_initial(V, np.zeros_like(V))
        g.step_barriers(16)
    assert small.sizes()[0] > 4096                  # the first capacity
    for a, b in zip(small.read_mesh(), large.read_mesh()):
        assert np.array_equal(a, b)
    assert np.array_equal(small.read_V(), large.read_V()) and np.array_equal(small.read_state(), large.read_state())
    small.close()
    large.close()


@pytest.mark.parametrize("precision", [32, 64])
def test_curved_run_does_not_depend_on_the_capacity(mdl, precision):
    """The factors of curved elements lie in groups of 32 elements: they keep their places when the
    arrays grow.  The context with room has been refined everywhere and coarsened to its roots before."""
    base = (24, 10, 2)
    p = W.lv_3d_q1_amr(base).replace(precision=precision, tau_refine=1e-12, tau_coarsen=1e-13, stimuli=[])
    xyz = [(i, j, k) for k in range(base[2]) for j in range(base[1]) for i in range(base[0])]
    small, large = mdl.Sim(p), mdl.Sim(p)
    peak = 0
    for eta in (1.0, 1.0, 0.0, 0.0):
        large.set_indicators(eta_s=np.full(large.sizes()[0], eta))
        large.step_barriers(1)
        peak = max(peak, large.sizes()[0])
    assert peak == 64 * len(xyz) and large.sizes()[0] == len(xyz)
    V = np.repeat(0.5 * (1.0 - np.tanh((np.array(xyz)[:, 0] - 12.0) / 2.0)), 8)
    for g in (small, large):
        g.set_initial(V, np.zeros_like(V))
        g.step_barriers(5)
    assert small.sizes()[0] > 4096
    for x, y in zip(small.read_mesh(), large.read_mesh()):
        assert np.array_equal(x, y)
    assert np.array_equal(small.read_V(), large.read_V()) and np.array_equal(small.read_state(), large.read_state())
    small.close()
    large.close()


@pytest.mark.parametrize("dim", [2, 3])
def test_small_adapting_fp32_default_sweep_matches_the_thread_sweep(mdl, dim):
    p = problem(dim, 1, 32, 1)
    a, b = mdl.Sim(p), mdl.Sim(p)
    b.set_sweep_variant(mdl.SWEEP_THREAD)
    a.step_barriers(60)
    b.step_barriers(60)
    assert np.array_equal(a.read_mesh()[1], b.read_mesh()[1])
    for x, y in ((a.read_V(), b.read_V()), (a.read_state(), b.read_state())):
        assert np.abs(x - y).max() <= 2e-5 * max(np.abs(y).max(), 1e-30)
    a.close()
    b.close()


@pytest.mark.parametrize("dim,order", [(2, 1), (2, 2), (3, 1), (3, 2)])
def test_launch_shapes_give_the_same_bits_on_a_small_mesh(mdl, dim, order):
    """The default's smaller blocks, and each shape that is set as it is set (a partial block)."""
    p = problem(dim, order, 32, 0)
    V = None
    for shape in (None, (64, 32), (128, 16), (256, 8)):
        g = mdl.Sim(p)
        if shape:
            g.set_tick_shape(*shape)
        g.step_barriers(3)
        V = g.read_V() if V is None else V
        assert np.array_equal(g.read_V(), V)
        g.close()

"""int V of FP32 contexts is an FP64 sum of the FP32 values with FP64 weights.

Tolerance: relative to sum |M V|.  A thread adds at most 28 values an element it visits, the block
and the partials' pass about 30 more sums, each within 2^-53 = 1.1e-16 of the partial sums so far, and
the weights carry 4 roundings: (28 n + 34) x 1.1e-16 = 6.9e-15 for one element a thread (n = 1), held
to 7e-15, and 3.2e-14 for nine.
"""
import math

import numpy as np
import pytest

import workloads as W
from oracle import basis
from tests.helpers import forest_arrays, random_forest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def mdl():
    import torch
    if not torch.cuda.is_available():
        pytest.fail("CUDA device required for -m gpu tests")
    from paper_2310_07607_gb300 import build, mdl as M
    build.build()
    return M


def problem(dim, order, base, extent, max_refine):
    return W.Problem(dim=dim, order=order, extent=extent, base=base, sigma_l=1.2, sigma_t=0.4, fibre=(0.6, 0.8, 0.0),
                     gamma=10.0 * order * order, dt_barrier=2.0 ** -10, max_refine=max_refine,
                     n_lts_levels=1, state_integrator=W.STATE_EXP, precision=32, amr_enabled=0, lts_enabled=0)


def check(g, prob, tol):
    V = g.read_V()
    level = g.read_mesh()[1].astype(int)
    h = [prob.extent[k] / (prob.base[k] * 2.0 ** np.arange(8)) for k in range(prob.dim)]
    m = np.prod([x / 2.0 for x in h], axis=0)[level][:, None] * basis.node_weights(prob.dim, prob.order)[None, :]
    t = m.reshape(-1) * V
    ref, scale = (math.fsum(t), math.fsum(np.abs(t))) if t.size < 10 ** 6 else (np.sum(t), np.sum(np.abs(t)))
    assert abs(g.stats()["integral_V"] - ref) <= tol * scale


@pytest.mark.parametrize("dim,order", [(2, 1), (2, 2), (3, 1), (3, 2)])
@pytest.mark.parametrize("field", ["rest", "front"])
def test_integral_of_fp32_contexts_is_an_fp64_sum(mdl, dim, order, field):
    base = (13, 11, 1) if dim == 2 else (7, 5, 3)
    prob = problem(dim, order, base, (1.3, 0.7, 0.37), 2)
    f = random_forest(dim, base, 2, prob.extent, steps=3, seed=5, tau=0.6)
    g = mdl.Sim(prob)
    g.upload_mesh(*forest_arrays(f))
    n = g.sizes()[1]
    rng = np.random.default_rng(7)
    V = np.full(n, 0.9371) if field == "rest" else 0.5 + 0.5 * np.sin(3.0 * np.arange(n) / n) + 0.01 * rng.uniform(size=n)
    g.set_initial(V, np.zeros(n))
    for _ in range(2):
        g.step_barriers(1)
        check(g, prob, 7e-15)
    g.close()


@pytest.mark.parametrize("dim,order,base", [(2, 2, (1672, 1664, 1)), (3, 2, (160, 136, 128))])
def test_integral_with_nine_elements_a_thread(mdl, dim, order, base):
    """2.78 M elements on 152 SMs of 2048 threads; resting tissue (a constant field), where the
    roundings of every thread are the same."""
    prob = problem(dim, order, base, (2.0, 1.7, 1.6), 0).replace(dt_barrier=2.0 ** -14)
    g = mdl.Sim(prob)
    n = g.sizes()[1]
    g.set_initial_f32(np.full(n, 0.9371, np.float32), np.zeros(n, np.float32))
    g.step_barriers(1)
    check(g, prob, 3.2e-14)
    g.close()

"""The cell reaction near its zeros.  I = (k u (u - a)(u - 1) + u w) / time scale vanishes exactly at
u = a, 1 (and 0) with w = 0 when each factor is formed by itself, so one long step leaves these values
bit for bit; and next to them its relative error stays a few roundings.

Tolerance next to the zeros (dt / time scale = 16): five roundings of I (2^-24 or 2^-53 each, relative)
times 16, and one rounding of the updated value.  Conductivities of 1e-25 mS/cm leave the operator out (1e-27 of
a step, below the rounding of every value used).
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


@pytest.mark.parametrize("dim,order,precision,integrator,variant,geometry", [
    (2, 1, 32, W.STATE_EXP, 0, 0), (2, 1, 32, W.STATE_EXP, 1, 0), (2, 1, 64, W.STATE_FE, 0, 0),
    (2, 1, 64, W.STATE_EXP, 1, 0), (2, 2, 32, W.STATE_EXP, 0, 0), (2, 2, 64, W.STATE_EXP, 0, 0),
    (3, 1, 32, W.STATE_EXP, 0, 0), (3, 2, 32, W.STATE_EXP, 0, 0), (3, 2, 32, W.STATE_FE, 0, 0),
    (3, 2, 32, W.STATE_EXP, 3, 0), (3, 2, 64, W.STATE_EXP, 0, 0), (3, 1, 32, W.STATE_EXP, 0, 1),
    (3, 1, 64, W.STATE_EXP, 0, 1)])
def test_reaction_keeps_its_zeros(mdl, dim, order, precision, integrator, variant, geometry):
    base = (8, 8, 1) if dim == 2 else (8, 4, 2)
    prob = W.Problem(dim=dim, order=order, extent=(1.0, 1.0, 1.0), base=base, sigma_l=1e-25, sigma_t=1e-25,
                     ionic_params=(8.0, 0.15, 0.002, 0.2, 0.3, 1.0 / 64), dt_barrier=0.25,
                     state_integrator=integrator, precision=precision)
    if geometry:
        prob = prob.replace(geometry=W.GEOMETRY_AFFINE, geo=(1.0, 0.1, 0, 0, 1.0, 0, 0, 0, 1.0, 0, 0, 0))
    dt = np.float32 if precision == 32 else np.float64
    a = float(dt(0.15))
    zeros = np.array([a, 1.0])
    near = np.concatenate([z + np.array([-1, 1])[:, None] * 2.0 ** -np.arange(6, 14) for z in (a, 1.0)]).reshape(-1)
    c = np.resize(np.concatenate([zeros, near]), prob.n_base).astype(dt).astype(np.float64)
    V0 = np.repeat(c, prob.n_p)
    g = mdl.Sim(prob)
    g.set_sweep_variant(variant)
    g.set_initial(V0, np.zeros_like(V0))
    g.step_barriers(1)
    V = g.read_V()
    assert np.array_equal(V[np.isin(V0, zeros)], V0[np.isin(V0, zeros)])
    # I from the exact differences (u - a, u - 1 of nearby numbers are exact); 16 = dt / time scale
    I = 8.0 * V0 * (V0 - a) * (V0 - 1.0)
    u = 2.0 ** -24 if precision == 32 else 2.0 ** -53
    assert np.all(np.abs(V - (V0 - 16.0 * I)) <= 16.0 * np.abs(I) * 5 * u + 2.0 * u * np.abs(V))
    g.close()

"""What this library is timed on: simulations as its users run them, over its public entry points.

A case names a kind of run, its base grid and how many barrier steps one pass takes.  The physics
(conductivities, element sizes, penalty, level counts, thresholds) are those of `workloads`; the
initial states are seeded developed fronts.  The kinds:

  plain     a small uniform FP64 square under global forward Euler, stepped and read back
  spiral    temporal adaptivity: a broken wave started afresh each pass, substeps by the cell's state
  slab      an adapting slab (2D or 3D, Q1 or Q2, FP32) carrying a planar wave, stepped and read back
  coupled   a uniform 3D Q2 FP32 block whose fields go to the host and come back each pass
  shell     an LV-like curved shell on its root mesh, FP32
  shellamr  the curved shell with octree adaptation, FP64
  batch     resident instances of mixed size, dimension and order, stepped together
  serve     a burst of small adapting requests through the serving loop, from admission to result
"""
import math

import numpy as np
import torch

import workloads as W
from paper_2310_07607_gb300 import mdl
from paper_2310_07607_gb300.serve import Request, Server


def listed():
    return [
        # the smallest resident run: 1024 Q1 elements in FP64, 1 ms of the 20 ms run per snapshot
        dict(name="plain2d_q1_fp64", kind="plain", n0=32, barriers=100),
        # spiral onset, 6400 Q1 elements, 5 levels of substeps, 1 ms per pass
        dict(name="spiral2d_q1", kind="spiral", n0=80, barriers=10),
        # the 2D slab: quadtree to depth 3, 4 levels, a snapshot every 20 barrier steps
        dict(name="slab2d_q1_amr", kind="slab", dim=2, order=1, n0=256, n1=256, n2=1, barriers=20),
        # a 2D request of the serving mix at its upper size, Q2, depth 2, 3 levels, oblique fibres
        dict(name="slab2d_q2_amr", kind="slab", dim=2, order=2, n0=181, n1=181, n2=1, barriers=20),
        # a 3D Q1 request of the serving mix, odd extents, depth 2, 3 levels, oblique fibres
        dict(name="slab3d_q1_amr", kind="slab", dim=3, order=1, n0=91, n1=32, n2=13, barriers=10),
        # the 3D slab (the benchmark's workload): octree to depth 3, 4 levels; the largest case
        dict(name="slab3d_q2_amr", kind="slab", dim=3, order=2, n0=128, n1=48, n2=20, barriers=4),
        # tissue coupled to a host model: fields uploaded, 4 barrier steps, fields read back
        dict(name="coupled3d_q2", kind="coupled", n0=61, n1=24, n2=20, barriers=4),
        # the LV-like shell, 184,320 curved Q1 elements, 4 levels
        dict(name="shell3d_q1", kind="shell", n0=240, n1=96, n2=8, barriers=8),
        # the adapting shell in FP64 (accuracy reference), depth 2, 4 levels
        dict(name="shell3d_q1_amr_fp64", kind="shellamr", n0=60, n1=24, n2=2, barriers=4),
        # 24 resident instances, 1e3 .. 1e5 elements each, half 2D Q1, half 3D Q1 / Q2
        dict(name="batch24_mixed", kind="batch", n0=24, barriers=8),
        # eight small adapting requests arriving at once, 2 ms each, served to completion
        dict(name="serve8_small", kind="serve", n0=8, horizon=2.0),
    ]


def draw(rng):
    def log(a, b):
        return int(round(math.exp(rng.uniform(math.log(a), math.log(b)))))

    kind = rng.choice(["plain", "spiral", "slab", "slab", "slab", "coupled", "shell", "shellamr", "batch", "serve"])
    if kind == "plain":
        return dict(kind=kind, n0=log(16, 128), barriers=log(20, 200))
    if kind == "spiral":
        return dict(kind=kind, n0=log(40, 160), barriers=log(4, 16))
    if kind == "slab":
        dim, order = rng.choice([(2, 1), (2, 2), (3, 1), (3, 2)])
        if dim == 2:
            return dict(kind=kind, dim=2, order=order, n0=log(24, 320), n1=log(24, 320), n2=1, barriers=log(8, 40))
        s = log(24, 120 if order == 1 else 110)
        return dict(kind=kind, dim=3, order=order, n0=s, n1=max(3, int(round(0.37 * s)) + rng.randint(-1, 1)),
                    n2=max(2, int(round(0.15 * s)) + rng.randint(-1, 1)), barriers=log(2, 10 if order == 1 else 4))
    if kind == "coupled":
        return dict(kind=kind, n0=log(9, 96), n1=log(5, 36), n2=log(3, 24), barriers=log(1, 8))
    if kind == "shell":
        return dict(kind=kind, n0=rng.randint(200, 280), n1=log(20, 110), n2=log(2, 10), barriers=log(2, 16))
    if kind == "shellamr":
        return dict(kind=kind, n0=log(24, 72), n1=log(10, 30), n2=log(2, 4), barriers=log(2, 6))
    if kind == "batch":
        return dict(kind=kind, n0=log(4, 24), barriers=log(2, 12))
    return dict(kind=kind, n0=log(2, 10), horizon=round(rng.uniform(0.5, 2.5), 3))


# --------------------------------------------------------------------------
# Problems.
# --------------------------------------------------------------------------

def _problem(case):
    k = case["kind"]
    if k == "plain":
        return W.scaled(W.plain_2d_q1_32x32(), (case["n0"], case["n0"], 1))
    if k == "spiral":
        return W.spiral_2d_q1(case["n0"])
    if k == "coupled":
        return W.scaled(W.slab_3d_q2(), (case["n0"], case["n1"], case["n2"])).replace(amr_enabled=0, max_refine=0)
    if k == "shell":
        p = W.lv_3d_q1((case["n0"], case["n1"], case["n2"]))
        # a coarser shell takes longer barrier steps: the substep that the cell state may ask for
        # grows with them, so that it stays within the 4 levels
        return p if case["n0"] >= 240 else p.replace(dt_bar_cell=0.016 * (240.0 / case["n0"]) ** 2)
    if k == "shellamr":
        return W.lv_3d_q1_amr((case["n0"], case["n1"], case["n2"])).replace(precision=64)
    dim, order, base = case["dim"], case["order"], (case["n0"], case["n1"], case["n2"])
    if (dim, order) == (2, 1):
        return W.scaled(W.slab_2d_q1_256(), base)
    if (dim, order) == (3, 2):
        return W.scaled(W.slab_3d_q2(), base)
    # the other two classes as the serving mix has them: element size, thresholds, fibres
    h = (0.0078125 if dim == 2 else 0.015625) * order
    ext = tuple(base[i] * h if i < dim else 1.0 for i in range(3))
    tau = W.SERVE_TAU[(dim, order)]
    return W.Problem(dim=dim, order=order, extent=ext, base=base, sigma_l=1.2, sigma_t=0.4,
                     fibre=W.fibre_from_angle(0.7), gamma=10.0 * order * order,
                     stimuli=[W.Stimulus((0.0, 0.0, 0.0), tuple(0.1 * e for e in ext), 1.0, 0.0, 1.0)],
                     dt_barrier=0.0, max_refine=2, n_lts_levels=3, tau_cell=0.5, tau_refine=tau[0], tau_coarsen=tau[1],
                     state_integrator=W.STATE_EXP, precision=32, amr_enabled=1, lts_enabled=1)


def _points(prob):
    """GL node coordinates of the root mesh in the library's order (roots x fastest)."""
    n1, d = prob.order + 1, prob.dim
    xi = np.array([-1.0, 1.0]) / math.sqrt(3.0) if n1 == 2 else np.array([-math.sqrt(0.6), 0.0, math.sqrt(0.6)])
    ax = [((np.arange(prob.base[k])[:, None] + 0.5 * (xi + 1.0)) * (prob.extent[k] / prob.base[k])) for k in range(d)]
    ne = prob.n_base
    X = np.empty((ne, n1 ** d, d))
    e, q = np.arange(ne), np.arange(n1 ** d)
    for k in range(d):
        X[:, :, k] = ax[k][(e % prob.base[k])[:, None], (q % n1)[None, :]]
        e, q = e // prob.base[k], q // n1
    return X.reshape(-1, d)


def _planar(prob, rng):
    """A wave travelling along x: its place, width and wake drawn from the seed."""
    x0 = prob.extent[0] * rng.uniform(0.4, 0.6)
    return W.planar_front_state(_points(prob), x0, rng.uniform(0.011, 0.013), rng.uniform(0.25, 0.35))


def _initial(case, prob, rng):
    if case["kind"] == "plain":
        r = prob.extent[0] * rng.uniform(0.3, 0.5)
        return W.front_state(_points(prob), (0.0, 0.0), r, rng.uniform(0.02, 0.03), rng.uniform(0.25, 0.35))
    if case["kind"] == "spiral":
        return W.spiral_state(_points(prob), prob.extent[0], rng.uniform(0.018, 0.022))
    if case["kind"] in ("shell", "shellamr"):
        # a surface of constant azimuth; the wave is wide against the coarse curved elements
        x0 = prob.extent[0] * rng.uniform(0.4, 0.6)
        return W.planar_front_state(_points(prob), x0, rng.uniform(0.09, 0.11), rng.uniform(0.5, 0.7))
    return _planar(prob, rng)


def _buffers(prob, n):
    """Host arrays for V and the state, n values each (page-locked in FP32): a program reads into them."""
    if prob.precision == 64:
        return [np.zeros(n), np.zeros(n)]
    return [torch.zeros(n, dtype=torch.float32, pin_memory=True).numpy() for _ in range(2)]


def _capacity(case, prob):
    """DOFs that a program makes room for: the mesh at full depth, or the roots and eight of their
    columns at full depth around the wave."""
    full = prob.n_base << (prob.dim * prob.max_refine)
    if case["kind"] == "slab":
        full = min(full, prob.n_base + 8 * (prob.n_base // prob.base[0] << (prob.dim * prob.max_refine)))
    return full * prob.n_p


# --------------------------------------------------------------------------
# Preparing and running.
# --------------------------------------------------------------------------

def _requests(case, rng):
    """Small requests of the four classes: 100 to 2000 base elements, depth 2, 3 levels."""
    out = []
    n = case["n0"]
    for i in range(n):
        ne = math.exp(math.log(100.0) + (math.log(2000.0) - math.log(100.0)) * (i + 0.5) / n)
        dim, order = ((2, 1), (3, 2), (2, 2), (3, 1))[i % 4]
        if dim == 2:
            side = int(round(math.sqrt(ne)))
            base, h = (side, side, 1), 8.0 * 0.0078125 * order
        else:
            s = (ne / 0.42) ** (1.0 / 3.0)
            base, h = tuple(max(2, int(round(f * s))) for f in (2.0, 0.7, 0.3)), 4.0 * 0.015625 * order
        ext = tuple(base[k] * h if k < dim else 1.0 for k in range(3))
        hi = tuple(rng.uniform(0.08, 0.12) * e for e in ext)
        tau = W.COMPLETED_TAU[(dim, order)]
        p = W.Problem(dim=dim, order=order, extent=ext, base=base, sigma_l=1.2, sigma_t=0.4,
                      fibre=W.fibre_from_angle(rng.uniform(0.0, math.pi)), gamma=10.0 * order * order,
                      stimuli=[W.Stimulus((0.0, 0.0, 0.0), hi, 1.0, 0.0, 1.0)], dt_barrier=0.0, max_refine=2,
                      n_lts_levels=3, tau_cell=0.5, tau_refine=tau[0], tau_coarsen=tau[1],
                      state_integrator=W.STATE_EXP, precision=32, amr_enabled=1, lts_enabled=1)
        out.append((p, case["horizon"]))
    return out


def prepare(case, seed):
    rng = np.random.default_rng(seed)
    kind = case["kind"]
    if kind == "serve":
        # the serving process: its loop is up, the requests arrive in `run`
        reqs = _requests(case, rng)
        bufs = [_buffers(p, _capacity(case, p)) for p, _ in reqs]

        def result(req, sim):
            V, s = bufs[req.rid]
            n = sim.read_fields_f32(V, s)[0].size
            return {"V": V, "s": s, "n": n, "lat": sim.read_activation().astype(np.float32)}

        return {"case": case, "server": Server(on_result=result), "requests": reqs}
    if kind == "batch":
        # resident instances, past the rounds in which the batch picks its launch shapes
        b = mdl.Batch()
        slots, bufs = [], []
        for p, _ in W.batch_instances(case["n0"], seed=4):
            V, s = _planar(p, rng)
            slots.append(b.admit(p, 1e6, V, s))
            bufs.append(_buffers(p, V.size))
        b.step(16)
        return {"case": case, "batch": b, "slots": slots, "bufs": bufs}
    prob = _problem(case)
    sim = mdl.Sim(prob)
    V, s = _initial(case, prob, rng)
    state = {"case": case, "sim": sim}
    if kind in ("spiral", "coupled"):
        state["start"] = _buffers(prob, V.size)
        state["start"][0][:], state["start"][1][:] = V, s
    else:
        sim.set_initial(V, s)
    if kind in ("slab", "shellamr"):
        sim.step_barriers(6)  # the adaptation reaches the wave's depth
    state["bufs"] = _buffers(prob, _capacity(case, prob))
    return state


def _read(state):
    sim = state["sim"]
    V, s = state["bufs"]
    if V.dtype == np.float64:
        n = sim.read_V(V).size
        sim.read_state(s)
    else:
        n = sim.read_fields_f32(V, s)[0].size
    return {"V": V, "s": s, "n": n}


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "serve":
        server = state["server"]
        reqs = [Request(i, p, h, 0.0) for i, (p, h) in enumerate(state["requests"])]
        server.done.clear()
        server.run(reqs, 0.0, drain=True)
        if any(r.rc for r in reqs):
            raise RuntimeError("a request failed: %s" % [r.rc for r in reqs])
        return [r.result for r in reqs]
    if kind == "batch":
        b = state["batch"]
        b.step(case["barriers"])
        out = []
        for slot, (V, s) in zip(state["slots"], state["bufs"]):
            out.append(b.slot(slot)[0].read_fields_f32(V, s))
        return out
    sim = state["sim"]
    if "start" in state:
        sim.set_initial_f32(*state["start"])
    sim.step_barriers(case["barriers"])
    return _read(state)


# --------------------------------------------------------------------------
# The work of a pass.
# --------------------------------------------------------------------------

# Bytes a DOF update cannot do without: its value and state read and written (twice the width on
# FP64), and the element's level, faces, neighbours and indicator sum over its DOFs.
def _bytes_per_update(prob):
    w = 4.0 * (2 if prob.precision == 64 else 1)
    n_p = (prob.order + 1) ** prob.dim
    per_elem = 36.0 if prob.dim == 2 else 44.0
    if prob.geometry:
        per_elem += w * (7 * n_p + 6 * 4 * 5)   # metric and mass per node, flux, area, penalty per face point
    return 4.0 * w + per_elem / n_p


def _updates_per_barrier(case, prob):
    """DOF updates of a barrier step: the DOFs of the (adapted) mesh times their substeps."""
    n_p = (prob.order + 1) ** prob.dim
    k = case["kind"]
    if k != "slab" and k != "shellamr":
        # substeps per element, as the levels of these meshes give them
        return n_p * prob.n_base * {"plain": 1.0, "spiral": 5.2, "coupled": 8.0, "shell": 2.1}[k]
    # an adapting mesh: the roots at one step, and the wave's band of root columns at full depth
    # and the finest substep
    cols = 1.3 if k == "shellamr" else {(2, 1): 3.2, (2, 2): 2.1, (3, 1): 0.11, (3, 2): 4.6}[(prob.dim, prob.order)]
    band = cols * prob.n_base / prob.base[0] * 2 ** (prob.dim * prob.max_refine)
    return n_p * (prob.n_base + band * 2 ** (prob.n_lts_levels - 1))


def work(case):
    k = case["kind"]
    if k == "batch":
        todo = [(p, p.n_base * p.n_p * 2.0 ** (p.n_lts_levels - 1) * case["barriers"])
                for p, _ in W.batch_instances(case["n0"], seed=4)]
    elif k == "serve":
        todo = [(p, 1.4 * p.n_base * p.n_p * h * 128.0 * p.order) for p, h in _requests(case, np.random.default_rng(0))]
    else:
        prob = _problem(case)
        todo = [(prob, _updates_per_barrier(case, prob) * case["barriers"])]
    # about 60 operations of the cell model and the indicator, and a line of the operator per direction
    return {"bytes": sum(_bytes_per_update(p) * u for p, u in todo),
            "flops": sum((60.0 + p.dim * 6.0 * (p.order + 1)) * u for p, u in todo)}


# --------------------------------------------------------------------------
# The same runs in 64 bits, in plain torch, on uniform grids.
# --------------------------------------------------------------------------

class _Uniform:
    """A box problem on its root mesh: dense SIPG blocks by quadrature, the Gershgorin levels and the
    level-by-level time stepping on a grid of elements."""

    def __init__(self, prob):
        d, p = prob.dim, prob.order
        self.prob, self.d, self.n1 = prob, d, p + 1
        n1 = self.n1
        x, w = np.polynomial.legendre.leggauss(n1)
        poly = [np.poly1d(np.poly([x[j] for j in range(n1) if j != i])) for i in range(n1)]
        poly = [q / q(x[i]) for i, q in enumerate(poly)]
        val = lambda s: np.array([q(s) for q in poly])            # noqa: E731
        der = lambda s: np.array([q.deriv()(s) for q in poly])    # noqa: E731
        h = [prob.extent[k] / prob.base[k] for k in range(d)]
        f = np.array(prob.fibre[:d]) / np.linalg.norm(prob.fibre)
        self.D = D = (prob.sigma_t * np.eye(d) + (prob.sigma_l - prob.sigma_t) * np.outer(f, f)) / (prob.chi * prob.cm)

        def kron(mats):   # node index a0 + n1 a1 + n1^2 a2: the last direction outermost
            out = np.ones((1, 1))
            for m in mats[::-1]:
                out = np.kron(out, m)
            return out

        eye, D1 = np.eye(n1), np.array([der(s) for s in x])
        grad = [kron([D1 * 2 / h[k] if j == k else eye for j in range(d)]) for k in range(d)]
        self.M = kron([np.diag(w) * h[k] / 2 for k in range(d)]).diagonal().copy()
        vol = sum(D[k, l] * grad[k].T @ np.diag(self.M) @ grad[l] for k in range(d) for l in range(d))
        self.own, self.nb = [], []
        for k in range(d):
            Wt = kron([np.diag(w) * h[j] / 2 if j != k else np.ones((1, 1)) for j in range(d)])
            kap = prob.gamma * D[k, k] / h[k]

            def trace(s, l=None):
                m = []
                for j in range(d):
                    if j == k:
                        m.append((der(s) * 2 / h[k] if l == k else val(s))[None, :])
                    else:
                        m.append(D1 * 2 / h[j] if l == j else eye)
                return kron(m)

            for s in (-1.0, 1.0):
                To, Tn = trace(s), trace(-s)
                Fo = s * sum(D[k, l] * trace(s, l) for l in range(d))
                Fn = s * sum(D[k, l] * trace(-s, l) for l in range(d))
                self.own.append(kap * To.T @ Wt @ To - 0.5 * To.T @ Wt @ Fo - 0.5 * Fo.T @ Wt @ To)
                self.nb.append(-kap * To.T @ Wt @ Tn - 0.5 * To.T @ Wt @ Fn + 0.5 * Fo.T @ Wt @ Tn)
        self.vol = vol
        # the CFL bound of every set of interior faces, the barrier step, and each element's level
        cfl = np.empty(1 << (2 * d))
        for c in range(cfl.size):
            L = (vol + sum(self.own[i] for i in range(2 * d) if c >> i & 1)) / self.M[:, None]
            cfl[c] = 1.0 / np.abs(L).sum(axis=1).max()
        self.B = prob.n_lts_levels - 1 if prob.lts_enabled else 0
        self.dt = prob.dt_barrier
        if self.dt <= 0:
            k = -20
            while 2.0 ** (-k - self.B) > cfl.min():
                k += 1
            self.dt = 2.0 ** -k
        dev = "cuda" if torch.cuda.is_available() else "cpu"
        shape = tuple(prob.base[:d][::-1])
        inside = np.zeros(shape, dtype=np.int64)
        for k in range(d):
            idx = np.arange(prob.base[k]).reshape([-1 if j == d - 1 - k else 1 for j in range(d)])
            inside = inside | ((idx > 0) * (1 << 2 * k)) | ((idx < prob.base[k] - 1) * (2 << 2 * k))
        lev = np.zeros(cfl.size, dtype=np.int64)
        if prob.lts_enabled:
            for c in range(cfl.size):
                while self.dt / 2.0 ** lev[c] > cfl[c]:
                    lev[c] += 1
        self.t = lambda a: torch.as_tensor(a, device=dev)  # noqa: E731
        self.bcfl, self.shape = self.t(lev[inside]), shape
        self.bcell = 0
        while prob.dt_bar_cell > 0 and self.dt / 2.0 ** self.bcell > prob.dt_bar_cell:
            self.bcell += 1
        X = _points(prob)
        self.stim = []
        for s in prob.stimuli:
            on = np.all([(X[:, k] >= s.lo[k] - 1e-12) & (X[:, k] <= s.hi[k] + 1e-12) for k in range(d)], axis=0)
            self.stim.append((self.t(on.reshape(shape + (-1,)).astype(np.float64)) * s.amplitude, s.t0, s.t1))
        self.tv, self.tM = self.t(vol), self.t(self.M)
        self.to, self.tn = [self.t(a) for a in self.own], [self.t(a) for a in self.nb]

    def residual(self, u):
        r = u @ self.tv.T
        for k in range(self.d):
            ax = self.d - 1 - k
            n = u.shape[ax]
            if n < 2:
                continue
            lo, hi = u.narrow(ax, 0, n - 1), u.narrow(ax, 1, n - 1)
            r.narrow(ax, 1, n - 1).add_(hi @ self.to[2 * k].T + lo @ self.tn[2 * k].T)
            r.narrow(ax, 0, n - 1).add_(lo @ self.to[2 * k + 1].T + hi @ self.tn[2 * k + 1].T)
        return r

    def current(self, t):
        return -sum((m for m, a, b in self.stim if a <= t < b), torch.zeros((), dtype=torch.float64, device=self.tM.device))

    def cell(self, V, w):
        k, a, e0, m1, m2, ts = self.prob.ionic_params
        vinf = -k * V * (V - a - 1)
        eps = e0 + m1 * w / torch.clamp(V + m2, min=1e-6)
        return (k * V * (V - a) * (V - 1) + V * w) / ts, eps, vinf, eps * (vinf - w) / ts

    def advance(self, V, w, barriers):
        """`barriers` barrier steps from t = 0 and a resting indicator."""
        V = self.t(np.asarray(V, np.float64)).reshape(self.shape + (-1,)).clone()
        w = self.t(np.asarray(w, np.float64)).reshape(self.shape + (-1,)).clone()
        eta = torch.zeros(self.shape, dtype=torch.float64, device=V.device)
        ts = self.prob.ionic_params[5]
        for n in range(barriers):
            b = torch.maximum(self.bcfl, (eta > self.prob.tau_cell) * self.bcell) if self.prob.lts_enabled else self.bcfl
            step = 2 ** (self.B - b)                      # ticks of an element's substep
            dte = (self.dt / 2.0 ** b.double())[..., None]
            old, acc, Ia, ga = V.clone(), torch.zeros_like(eta), None, None
            for i in range(1 << self.B):
                due = (i % step == 0)[..., None]
                th = ((i % step).double() / step)[..., None]
                seen = torch.where(due, V, old + th * (V - old))
                t = (n * 2 ** self.B + i) * (self.dt / 2 ** self.B)
                so = self.current(t)
                I, eps, vinf, g = self.cell(V, w)
                I = I + so
                if i == 0:
                    Ia, ga = I, g
                un = V + dte * (-self.residual(seen) / self.tM - I)
                x = -eps * dte / ts
                wn = vinf + (w - vinf) * torch.exp(x) if self.prob.state_integrator else w + dte * g
                sm = torch.zeros_like(V)
                for m, a, c in self.stim:
                    tm = t + 0.5 * dte
                    sm = sm - m * ((tm >= a) & (tm < c))
                Im, _, _, gm = self.cell(0.5 * (V + un), 0.5 * (w + wn))
                term = (self.tM * ((Im + sm - Ia) ** 2 + (gm - ga) ** 2)).sum(-1)
                acc = torch.where(due[..., 0], acc + dte[..., 0] * term, acc)
                old = torch.where(due, V, old)
                V, w = torch.where(due, un, V), torch.where(due, wn, w)
            eta = torch.sqrt(acc) / self.dt
        return V.reshape(-1), w.reshape(-1)


def exact(case, seed):
    kind = case["kind"]
    rng = np.random.default_rng(seed)
    if kind == "batch":
        out = []
        for p, _ in W.batch_instances(case["n0"], seed=4):
            V, s = _planar(p, rng)
            out.append(_Uniform(p).advance(V, s, 16 + case["barriers"]))
        return out
    if kind not in ("plain", "spiral", "coupled"):
        return None   # adapting and curved meshes: no uniform grid to restate them on
    prob = _problem(case)
    V, s = _initial(case, prob, rng)
    if prob.precision == 32 and kind in ("spiral", "coupled"):
        V, s = V.astype(np.float32), s.astype(np.float32)
    V, s = _Uniform(prob).advance(V, s, case["barriers"])
    return {"V": V, "s": s, "n": None}

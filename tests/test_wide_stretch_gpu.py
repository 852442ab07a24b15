"""Double-word handles at large stretches and rotations: their bonds stay in double-word
arithmetic up to |y|^2 / |xi|^2 = 1 +- 1/2, so that a strained or rotated body costs what a
resting one does, and within the error of that arithmetic.

One step from v = 0 against the oracle, in units of c V_j of each bond: the oracle's s (and
that of the bonds past the range) carries 8 2^-53; num = eta . (2 xi + eta) carries 2^-44.6
of its terms, at most |eta| (|xi| + |y|), which is 2^-44.6 |eta| / |xi| of s; the rest of the
bond 2^-44 s, the sums (segments of 16, double-words) 2^-43 s: in all
8 2^-53 + 2^-44 |eta| / |xi| + 2^-42 |s|."""
import time

import numpy as np
import pytest

import oracle
import paper_2105_04150_gb300 as pdgb
import workloads

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _need_gpu():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    pdgb.build()
    oracle.build()


def _state(shape, strain, angle, jitter=0.0):
    w = workloads.tensile_bar(*shape, rate=0.0, sc=5.0)
    rng = np.random.default_rng(5)
    w.bc_type[:] = 0
    if jitter:
        w.coords = w.coords + rng.uniform(-jitter, jitter, w.coords.shape) * w.dx
        w.volumes = w.volumes * rng.uniform(0.5, 2.0, w.n)
    c, s = np.cos(angle), np.sin(angle)
    R = np.array([[c, -s, 0], [s, c, 0], [0, 0, 1.0]])
    A = np.eye(3) + strain * (np.eye(3) + rng.uniform(-0.2, 0.2, (3, 3)))
    x = w.coords - w.coords.mean(0)
    return w, x @ A.T @ R.T - x + rng.uniform(-0.05, 0.05, (w.n, 3)) * strain * w.dx


STATES = [(1e-3, 0.0), (7.9e-3, 0.0), (0.05, 0.0), (0.2, 0.0), (0.24, 0.0), (-0.1, 0.0),
          (-0.28, 0.0), (-0.5, 0.0), (0.5, 0.0), (1e-4, 0.3), (0.1, 1.5)]


@pytest.mark.parametrize("strain,angle", STATES)
@pytest.mark.parametrize("jitter", [0.0, 0.2])
def test_bond_based_step(strain, angle, jitter):
    w, u = _state((11, 8, 7), strain, angle, jitter)
    off, idx = oracle.cut_family(w.coords, w.horizon, w.cuts_array())
    om = oracle.Model.from_workload(w, off, idx)
    uo, vo, mu = u.copy(), np.zeros((w.n, 3)), om.fresh_bonds()
    om.run(0, 1, uo, vo, mu)
    m = pdgb.Model.from_workload(w, precision=pdgb.PD_PREC_DW)
    m.set_state(u, np.zeros((w.n, 3)), 0)
    m.step(1)
    _, vg = m.state()
    m.close()
    c = oracle.micromodulus(w.bulk_modulus, w.horizon)
    rows = np.repeat(np.arange(w.n), np.diff(off))
    xi, eta = w.coords[idx] - w.coords[rows], u[idx] - u[rows]
    L = np.linalg.norm(xi, axis=1)
    s = np.abs(np.linalg.norm(xi + eta, axis=1) / L - 1.0)
    e = np.linalg.norm(eta, axis=1) / L
    tol = np.bincount(rows, w.volumes[idx] * (8 * 2.0 ** -53 + 2.0 ** -44 * e + 2.0 ** -42 * s),
                      minlength=w.n)
    tol = tol * c * w.dt / w.density + 4 * 2.0 ** -53 * np.abs(vo).max(1)
    assert (np.abs(vg - vo).max(1) <= tol).all()


@pytest.mark.parametrize("strain,angle", STATES)
@pytest.mark.parametrize("jitter", [0.0, 0.2])
def test_state_based_step(strain, angle, jitter):
    # the same error of e / |xi| of each bond, and through it of theta: as in the state-based
    # step's test, with the bond's error in place of its 16 2^-53 and 2^-44 s
    w, u = _state((11, 8, 7), strain, angle, jitter)
    K = w.bulk_modulus
    G = 0.6 * K
    w.state_based = (K, G)
    off, idx = oracle.cut_family(w.coords, w.horizon, w.cuts_array())
    om = oracle.Model.from_workload(w, off, idx)
    uo, vo, mu = u.copy(), np.zeros((w.n, 3)), om.fresh_bonds()
    om.run(0, 1, uo, vo, mu)
    m = pdgb.Model.from_workload(w, precision=pdgb.PD_PREC_DW)
    m.set_state(u, np.zeros((w.n, 3)), 0)
    m.step(1)
    _, vg = m.state()
    m.close()
    rows = np.repeat(np.arange(w.n), np.diff(off))
    xi, eta = w.coords[idx] - w.coords[rows], u[idx] - u[rows]
    L = np.linalg.norm(xi, axis=1)
    s = np.abs(np.linalg.norm(xi + eta, axis=1) / L - 1.0).max()
    e = (np.linalg.norm(eta, axis=1) / L).max()
    mv = np.bincount(rows, L * L * w.volumes[idx], minlength=w.n)
    ds = 16 * 2.0 ** -53 + 2.0 ** -44 * e + 2.0 ** -42 * s      # both sides' error of e / |xi|
    dth = 3 * ds + 300 * 2.0 ** -53 * 3 * s
    per = (3 * K + 5 * G) * dth + 15 * G * ds + 300 * 2.0 ** -53 * (3 * (3 * K + 5 * G) + 15 * G) * s
    tol = np.bincount(rows, w.volumes[idx] * L * (1 / mv[rows] + 1 / mv[idx]), minlength=w.n) * per
    tol = tol * w.dt / w.density + 4 * 2.0 ** -53 * np.abs(vo).max(1)
    assert (np.abs(vg - vo).max(1) <= tol).all()


def _ratio(run, limit):
    """Largest time of run[1:] over that of run[0], the least of up to 12 turns each, in turn,
    until it is within the limit (others may use the device)."""
    best = [float("inf")] * len(run)
    for _ in range(12):
        for k, r in enumerate(run):
            best[k] = min(best[k], r())
        if _ >= 2 and max(best[1:]) <= limit * best[0]:
            break
    return max(best[1:]) / best[0]


@pytest.mark.parametrize("state_based", [False, True])
def test_a_strained_or_turned_body_costs_what_a_resting_one_does(state_based):
    # (all of its bonds in FP64 would take 6 to 9 times as long)
    runs, models = [], []
    for strain, angle in ((1e-4, 0.0), (2e-2, 0.0), (0.15, 0.0), (2e-2, 0.5)):
        w, u = _state((120, 25, 25), strain, angle)
        if state_based:
            w.state_based = (w.bulk_modulus, 0.6 * w.bulk_modulus)
        m = pdgb.Model.from_workload(w, precision=pdgb.PD_PREC_DW)
        models.append(m)

        def run(m=m, u=u):
            m.set_state(u, np.zeros_like(u), 0)
            m.step(2)
            m.sync()
            t = time.perf_counter()
            m.step(6)
            m.sync()
            return time.perf_counter() - t
        runs.append(run)
    assert _ratio(runs, 1.5) <= 1.5
    for m in models:
        m.close()


def test_the_reverse_sweep_of_a_strained_body_costs_what_a_resting_one_does():
    runs, models = [], []
    for strain, angle in ((1e-4, 0.0), (2e-2, 0.0), (2e-2, 0.5)):
        w, u = _state((100, 40, 4), strain, angle)
        m = pdgb.Model.from_workload(w, precision=pdgb.PD_PREC_DW)
        models.append(m)
        g = np.random.default_rng(0).normal(size=u.shape)

        def run(m=m, u=u, g=g):
            m.set_state(u, np.zeros_like(u), 0)
            pdgb.pd_adjoint_forward(m.h, 40)
            m.sync()
            t = time.perf_counter()
            pdgb.pd_adjoint_backward(m.h, g, None, want_c=False)
            return time.perf_counter() - t
        runs.append(run)
    assert _ratio(runs, 1.5) <= 1.5
    for m in models:
        m.close()

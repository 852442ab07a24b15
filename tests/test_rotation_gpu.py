"""FP64 steps of a rotated body against the exact step: the error has to stay that of the
literal FP64 form at every angle.

One step from a given state with v = 0, so that v = dt F / rho, against the same sums in
long double (at least 64 bits).  The literal form rounds s = |y| / |xi| - 1 of a bond as
follows, in units of u = 2^-53, each rounding uniform in half an ulp and so at most
u / sqrt(3) rms of the rounded value: xi_c, eta_c and y_c, at most |xi|, 2 |xi| and |y| in
size, give sqrt(1 + 4 + 1) / sqrt(3) = 1.4 of |y|; the products and sums of |y|^2 half of
three, 0.5; 1/|y| after Newton's steps and the stored 1/|xi| at most 1 each; |y| 0.6.  In
quadrature 2.2 u rms.  Bonds' errors are independent (the nodes are moved off the lattice
at random), so the rms over all nodes and components of the force's error is at most that
of sum_j c V_j 2.2 u y_c / |y|.  The state-based force has it in each bond's e and, through
the dilation, in theta_i and theta_j."""
import numpy as np
import pytest

import oracle
import paper_2105_04150_gb300 as pdgb
import workloads

pytestmark = pytest.mark.gpu

ANGLES = [0.004, 0.012, 0.03, 0.1, 0.3, 1.5]
RMS_S = 2.2 * 2.0 ** -53


@pytest.fixture(scope="module", autouse=True)
def _need_gpu():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    pdgb.build()
    oracle.build()


def _rotated(angle, volumes_vary):
    w = workloads.tensile_bar(14, 9, 8, rate=0.0, sc=0.5)
    rng = np.random.default_rng(11)
    w.bc_type[:] = 0
    w.coords = w.coords + rng.uniform(-0.2, 0.2, w.coords.shape) * w.dx
    if volumes_vary:
        w.volumes = w.volumes * rng.uniform(0.5, 2.0, w.n)
    axis = np.array([2.0, -1.0, 2.0]) / 3.0
    K = np.array([[0, -axis[2], axis[1]], [axis[2], 0, -axis[0]], [-axis[1], axis[0], 0]])
    R = np.eye(3) + np.sin(angle) * K + (1 - np.cos(angle)) * K @ K
    x = w.coords - w.coords.mean(0)
    u = (x + 1e-4 * x @ rng.uniform(-1, 1, (3, 3)).T) @ R.T - x
    off, idx = oracle.cut_family(w.coords, w.horizon, w.cuts_array())
    rows = np.repeat(np.arange(w.n), np.diff(off))
    ld = np.longdouble
    xi = w.coords[idx].astype(ld) - w.coords[rows].astype(ld)
    y = xi + (u[idx].astype(ld) - u[rows].astype(ld))
    L, r = np.sqrt((xi * xi).sum(1)), np.sqrt((y * y).sum(1))
    return w, u, rows, idx, L, r, y / r[:, None]


def _force(w, u):
    m = pdgb.Model.from_workload(w, precision=pdgb.PD_PREC_F64)
    m.set_state(u, np.zeros((w.n, 3)), 0)
    m.step(1)
    _, v = m.state()
    m.close()
    return v * (w.density / w.dt)


def _add(rows, n, terms):
    out = np.zeros((n,) + terms.shape[1:], terms.dtype)
    np.add.at(out, rows, terms)
    return out


def _rms(a):
    return float(np.sqrt(np.mean(np.asarray(a, np.float64) ** 2)))


@pytest.mark.parametrize("volumes_vary", [False, True])
@pytest.mark.parametrize("angle", ANGLES)
def test_bond_based_step_of_a_rotated_body(angle, volumes_vary):
    w, u, rows, idx, L, r, d = _rotated(angle, volumes_vary)
    c = oracle.micromodulus(w.bulk_modulus, w.horizon)
    cV = c * w.volumes[idx]
    exact = _add(rows, w.n, (cV * (r / L - 1))[:, None] * d)
    got = _force(w, u)
    d2 = np.asarray(d, np.float64) ** 2
    bound = RMS_S * _rms(np.sqrt(_add(rows, w.n, (cV ** 2)[:, None] * d2)))
    assert np.abs(np.asarray(exact, np.float64)).max() > 0
    assert _rms(got - exact) <= bound


@pytest.mark.parametrize("volumes_vary", [False, True])
@pytest.mark.parametrize("angle", ANGLES)
def test_state_based_step_of_a_rotated_body(angle, volumes_vary):
    w, u, rows, idx, L, r, d = _rotated(angle, volumes_vary)
    K = w.bulk_modulus
    G = 0.6 * K
    w.state_based = (K, G)
    V = w.volumes[idx]
    e = r - L
    m = _add(rows, w.n, L * L * V)
    th = 3 * _add(rows, w.n, L * e * V) / m
    beta = 15 * G / m
    alpha = 3 * K * th / m - beta * th / 3
    t = (alpha[rows] + alpha[idx]) * L + (beta[rows] + beta[idx]) * e
    exact = _add(rows, w.n, (t * V)[:, None] * d)
    got = _force(w, u)
    # rms of the error: each bond's e, then theta_j of the neighbours, then theta_i
    f64 = lambda a: np.asarray(a, np.float64)
    L, m, d = f64(L), f64(m), f64(d)
    dth = 3 * RMS_S / m * np.sqrt(_add(rows, w.n, (L * L * V) ** 2))
    k = abs(3 * K - 5 * G)
    own = ((beta[rows] + beta[idx]) * L * RMS_S * V)
    own = np.sqrt(_add(rows, w.n, f64(own)[:, None] ** 2 * d ** 2))
    nb = np.sqrt(_add(rows, w.n, (k / m[idx] * dth[idx] * L * V)[:, None] ** 2 * d ** 2))
    ni = np.abs(_add(rows, w.n, (L * V)[:, None] * d)) * (k / m * dth)[:, None]
    bound = _rms(own) + _rms(nb) + _rms(ni)
    assert np.abs(f64(exact)).max() > 0
    assert _rms(got - exact) <= bound

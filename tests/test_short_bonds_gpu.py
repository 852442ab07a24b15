"""FP64 steps of a body with bonds far shorter than its longest: their error has to stay that
of the literal FP64 form, relative to each bond's own length.

A lattice moved off itself with close partners to some of its nodes, one step from v = 0
against the same sums in long double; the literal form's rms error of a bond's s is at
most 2.2 2^-53 whatever its length (test_rotation_gpu.py derives it: differences of close
numbers are exact), of a node's force that of sum_j c V_j 2.2 2^-53 y / |y|."""
import numpy as np
import pytest

import oracle
import paper_2105_04150_gb300 as pdgb
import workloads

pytestmark = pytest.mark.gpu

RMS_S = 2.2 * 2.0 ** -53


@pytest.fixture(scope="module", autouse=True)
def _need_gpu():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    pdgb.build()
    oracle.build()


def _add(rows, n, terms):
    out = np.zeros((n,) + terms.shape[1:], terms.dtype)
    np.add.at(out, rows, terms)
    return out


@pytest.mark.parametrize("gap", [0.3, 0.03, 1e-3, 1e-5, 1e-8])
@pytest.mark.parametrize("strain", [1e-4, 6e-3])
@pytest.mark.parametrize("state_based", [False, True])
def test_close_pairs(gap, strain, state_based):
    w = workloads.tensile_bar(10, 7, 6, rate=0.0, sc=0.5)
    rng = np.random.default_rng(13)
    x = w.coords + rng.uniform(-0.2, 0.2, w.coords.shape) * w.dx
    pick = rng.choice(len(x), 90, replace=False)
    d = rng.normal(size=(90, 3))
    x = np.concatenate([x, x[pick] + gap * w.dx * d / np.linalg.norm(d, axis=1)[:, None]])
    n = len(x)
    w.coords, w.volumes = x, w.dx ** 3 * rng.uniform(0.5, 2.0, n)
    w.bc_type, w.bc_disp, w.bc_force = np.zeros((n, 3), np.uint8), np.zeros((n, 3)), np.zeros((n, 3))
    K = w.bulk_modulus
    G = 0.6 * K
    if state_based:
        w.state_based = (K, G)
    u = strain * (x - x.mean(0)) @ (np.eye(3) + rng.uniform(-0.1, 0.1, (3, 3))).T
    off, idx = oracle.cut_family(w.coords, w.horizon, w.cuts_array())
    rows = np.repeat(np.arange(n), np.diff(off))
    ld = np.longdouble
    xi = x[idx].astype(ld) - x[rows].astype(ld)
    y = xi + (u[idx].astype(ld) - u[rows].astype(ld))
    L, r = np.sqrt((xi * xi).sum(1)), np.sqrt((y * y).sum(1))
    d = y / r[:, None]
    V = w.volumes[idx]
    m = pdgb.Model.from_workload(w, precision=pdgb.PD_PREC_F64)
    m.set_state(u, np.zeros((n, 3)), 0)
    m.step(1)
    got = m.state()[1] * (w.density / w.dt)
    m.close()
    f64 = lambda a: np.asarray(a, np.float64)
    if not state_based:
        cV = oracle.micromodulus(K, w.horizon) * V
        exact = _add(rows, n, (cV * (r / L - 1))[:, None] * d)
        rms = RMS_S * np.sqrt(_add(rows, n, (cV ** 2)[:, None] * f64(d) ** 2))
    else:
        e = r - L
        mv = _add(rows, n, L * L * V)
        th = 3 * _add(rows, n, L * e * V) / mv
        beta = 15 * G / mv
        alpha = 3 * K * th / mv - beta * th / 3
        t = (alpha[rows] + alpha[idx]) * L + (beta[rows] + beta[idx]) * e
        exact = _add(rows, n, (t * V)[:, None] * d)
        L, mv, d, beta = f64(L), f64(mv), f64(d), f64(beta)
        dth = 3 * RMS_S / mv * np.sqrt(_add(rows, n, (L * L * V) ** 2))
        k = abs(3 * K - 5 * G)
        own = np.sqrt(_add(rows, n, ((beta[rows] + beta[idx]) * L * RMS_S * V)[:, None] ** 2 * d ** 2))
        nb = np.sqrt(_add(rows, n, (k / mv[idx] * dth[idx] * L * V)[:, None] ** 2 * d ** 2))
        ni = np.abs(_add(rows, n, (L * V)[:, None] * d)) * (k / mv * dth)[:, None]
        rms = own + nb + ni
    # the nodes with a close partner, where that bond's error would show
    near = np.concatenate([pick, np.arange(n - 90, n)])
    err = f64(got - exact)[near]
    assert np.sqrt(np.mean(err ** 2)) <= np.sqrt(np.mean(rms[near] ** 2))

"""FP64 step of a body of many horizons in length: the error at its origin, where the FP64
coordinates are fine, has to stay that of the literal FP64 form.

The positions of the three-word records lie on one grid, that of the largest coordinate.
One step from v = 0 of a line of nodes moved off their lattice, the force of the nodes near
the origin against the same sums in long double; the literal form's rms error of a bond's
s is at most 2.2 2^-53 (test_rotation_gpu.py derives it), of the node's force that of
sum_j c V_j 2.2 2^-53 y / |y|."""
import time

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


def _body(n):
    w = workloads.tensile_bar(n, 1, 1, rate=0.0, sc=0.5)
    rng = np.random.default_rng(12)
    w.bc_type[:] = 0
    w.coords = w.coords.copy()
    w.coords[:, 0] += rng.uniform(-0.2, 0.2, n) * w.dx
    return w


def _near(w, u, k):
    """The first k nodes' bonds in long double: rows, neighbours, L, r and direction."""
    off, idx = oracle.cut_family(w.coords, w.horizon, w.cuts_array())
    idx, rows = idx[:off[k]], np.repeat(np.arange(k), np.diff(off[:k + 1]))
    ld = np.longdouble
    xi = w.coords[idx, 0].astype(ld) - w.coords[rows, 0].astype(ld)
    y = xi + (u[idx, 0].astype(ld) - u[rows, 0].astype(ld))
    return rows, idx, np.abs(xi), np.abs(y), np.sign(y)


@pytest.mark.parametrize("n", [2000, 20000, 200000])
@pytest.mark.parametrize("strain", [1e-4, 1e-3, 7e-3, -7e-3])
def test_force_near_the_origin(n, strain):
    w = _body(n)
    k = 400
    u = np.zeros((n, 3))
    u[:, 0] = strain * w.coords[:, 0]
    rows, idx, L, r, d = _near(w, u, k)
    c = oracle.micromodulus(w.bulk_modulus, w.horizon)
    cV = c * w.volumes[idx]
    exact = np.zeros(k, np.longdouble)
    np.add.at(exact, rows, cV * (r / L - 1) * d)
    m = pdgb.Model.from_workload(w, precision=pdgb.PD_PREC_F64)
    m.set_state(u, np.zeros((n, 3)), 0)
    m.step(1)
    _, v = m.state()
    m.close()
    err = np.asarray(v[:k, 0] * (w.density / w.dt) - exact, np.float64)
    bound = RMS_S * np.sqrt(np.mean(np.bincount(rows, cV ** 2, minlength=k)))
    assert np.sqrt(np.mean(err ** 2)) <= bound


@pytest.mark.parametrize("n", [2000, 200000])
@pytest.mark.parametrize("strain", [1e-3, 7e-3])
def test_stiffness_gradient_near_the_origin(n, strain):
    # dL/dc = dt/rho s V_j (y/|y|).w with w = gv: s to 2.2 2^-53 rms, the products to 4 2^-53
    # of themselves
    w = _body(n)
    k = 400
    u = np.zeros((n, 3))
    u[:, 0] = strain * w.coords[:, 0]
    rows, idx, L, r, d = _near(w, u, k)
    gv = np.zeros((n, 3))
    gv[:, 0] = 1.0 + 0.5 * np.sin(np.arange(n))
    m = pdgb.Model.from_workload(w, precision=pdgb.PD_PREC_F64)
    m.set_state(u, np.zeros((n, 3)), 0)
    pdgb.pd_adjoint_forward(m.h, 1)
    gc, _, _, _ = pdgb.pd_adjoint_backward(m.h, np.zeros((n, 3)), gv)
    m.close()
    f = w.dt / w.density * w.volumes[idx] * gv[rows, 0]
    s = r / L - 1
    err = np.asarray(gc[:len(rows)] - f * s * d, np.float64) / f
    assert np.sqrt(np.mean(err ** 2)) <= RMS_S + 4 * 2.0 ** -53 * abs(strain)


@pytest.mark.parametrize("offset", [(1e6, 1e6, 1e6), (-3e5, 0.0, 0.0), (0.0, 5e7, 2e3)])
@pytest.mark.parametrize("batch", [False, True])
def test_a_body_far_from_the_origin(offset, batch):
    # a body of ordinary length anywhere (offsets in spacings): the same cost and, against the
    # sums with its own coordinates in long double, the same bound
    runs, models = [], []
    for off3 in ((0.0, 0.0, 0.0), offset):
        w = workloads.tensile_bar(100, 20, 20, rate=0.0, sc=0.5)
        rng = np.random.default_rng(12)
        w.bc_type[:] = 0
        w.coords = w.coords + rng.uniform(-0.2, 0.2, w.coords.shape) * w.dx + np.array(off3) * w.dx
        A = 2e-3 * (np.eye(3) + rng.uniform(-0.2, 0.2, (3, 3)))
        u = (w.coords - w.coords.mean(0)) @ A.T
        if batch:
            m = pdgb.Model.batch([w], precision=pdgb.PD_PREC_F64)
        else:
            m = pdgb.Model.from_workload(w, precision=pdgb.PD_PREC_F64)
        models.append(m)
        m.set_state(u, np.zeros_like(u), 0)
        m.step(1)
        got = m.state()[1] * (w.density / w.dt)

        def run(m=m, u=u):
            m.set_state(u, np.zeros_like(u), 0)
            m.step(2)
            m.sync()
            s = time.perf_counter()
            m.step(10)
            m.sync()
            return time.perf_counter() - s
        runs.append(run)
    here = far = float("inf")
    for k in range(12):     # the least of up to 12 turns each (others may use the device)
        here, far = min(here, runs[0]()), min(far, runs[1]())
        if k >= 2 and far <= 1.5 * here:
            break
    for m in models:
        m.close()
    off, idx = oracle.cut_family(w.coords, w.horizon, w.cuts_array())
    rows = np.repeat(np.arange(w.n), np.diff(off))
    ld = np.longdouble
    xi = w.coords[idx].astype(ld) - w.coords[rows].astype(ld)
    y = xi + (u[idx].astype(ld) - u[rows].astype(ld))
    L, r = np.sqrt((xi * xi).sum(1)), np.sqrt((y * y).sum(1))
    d = y / r[:, None]
    cV = oracle.micromodulus(w.bulk_modulus, w.horizon) * w.volumes[idx]
    exact, var = np.zeros((w.n, 3), ld), np.zeros((w.n, 3))
    np.add.at(exact, rows, (cV * (r / L - 1))[:, None] * d)
    np.add.at(var, rows, (cV ** 2)[:, None] * np.asarray(d, np.float64) ** 2)
    err = np.asarray(got - exact, np.float64)
    assert np.sqrt(np.mean(err ** 2)) <= RMS_S * np.sqrt(np.mean(var))
    assert far <= 1.5 * here

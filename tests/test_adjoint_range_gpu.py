"""The reverse sweep over the whole range of FP64: a seed on one node whose influence decays
by orders of magnitude from horizon to horizon, and seeds that are denormal numbers.

A majorant of the sweep bounds both sides' rounding: with every |K d| <= 2 c / L
(V_m |w_j| + V_j |w_m|) and sums of absolute values, the FP64 sweep errs by at most
200 2^-53 of the majorant a step (a dozen operations a bond and the sum), the double-word
one by 2^-40 (2^-44 a term and 122 sums of 2^-47).  dL/dc = dt/rho s V_j (y/|y|).w, the
oracle's s to 8 2^-53.  A denormal number adds half of 2^-1074 an operation."""
import numpy as np
import pytest

import oracle
import paper_2105_04150_gb300 as pdgb
import workloads

pytestmark = pytest.mark.gpu

N = 12


@pytest.fixture(scope="module", autouse=True)
def _need_gpu():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    pdgb.build()
    oracle.build()


@pytest.mark.parametrize("volumes_vary", [False, True])
@pytest.mark.parametrize("seed_scale", [1.0, 1e-60, 1e50])
@pytest.mark.parametrize("precision", [pdgb.PD_PREC_F64, pdgb.PD_PREC_DW])
def test_far_from_the_seed(precision, seed_scale, volumes_vary):
    w = workloads.tensile_bar(40, 3, 2, rate=0.0, sc=0.5)
    w.bc_type[:] = 0
    w.dt = 1e-9
    rng = np.random.default_rng(8)
    if volumes_vary:
        w.volumes = w.volumes * rng.uniform(0.5, 2.0, w.n)
    u0 = 1e-3 * (w.coords - w.coords.mean(0)) + rng.uniform(-1, 1, (w.n, 3)) * 1e-4 * w.dx
    v0 = np.zeros((w.n, 3))
    off, idx = oracle.cut_family(w.coords, w.horizon, w.cuts_array())
    c = oracle.micromodulus(w.bulk_modulus, w.horizon)
    gu, gv = np.zeros((w.n, 3)), np.zeros((w.n, 3))
    gu[0] = np.array([0.3, -0.5, 0.8]) * seed_scale
    om = oracle.Model.from_workload(w, off, idx, c=c)
    gc_o, _, gu_o, gv_o = oracle.adjoint(om, 0, N, u0, v0, om.fresh_bonds(), gu, gv)
    m = pdgb.Model.from_workload(w, precision=precision, c=c)
    m.set_state(u0, v0, 0)
    pdgb.pd_adjoint_forward(m.h, N)
    gc, _, gu0, gv0 = pdgb.pd_adjoint_backward(m.h, gu, gv)
    m.close()
    rows = np.repeat(np.arange(w.n), np.diff(off))
    xi = w.coords[idx] - w.coords[rows]
    L = np.linalg.norm(xi, axis=1)
    s = 2 * np.abs(np.linalg.norm(xi + u0[idx] - u0[rows], axis=1) / L - 1.0)  # (12 short steps)
    dr = w.dt / w.density
    eps = 200 * 2.0 ** -53 if precision == pdgb.PD_PREC_F64 else 2.0 ** -40
    au, av = np.abs(gu).sum(1), np.abs(gv).sum(1)
    tolc = np.zeros(len(idx))
    for n in range(N):
        ww = av + w.dt * au
        tolc += dr * w.volumes[idx] * ww[rows] * (8 * 2.0 ** -53 + (2.0 ** -44 + (n + 1) * eps) * s)
        au = au + dr * np.bincount(rows, 2 * c / L * (w.volumes[rows] * ww[idx] + w.volumes[idx] * ww[rows]),
                                   minlength=w.n)
        av = ww
    tiny = 1000 * N * 2.0 ** -1074
    reached = np.abs(gu_o).max(1)
    assert 0 < reached[reached > 0].min() < 1e-30 * reached.max()   # the range is used
    assert 0 < np.abs(gc_o[gc_o != 0]).min() < 1e-30 * np.abs(gc_o).max()
    assert (np.abs(gu0 - gu_o).max(1) <= N * eps * au + tiny).all()
    assert (np.abs(gv0 - gv_o).max(1) <= N * eps * av + tiny).all()
    assert (np.abs(gc - gc_o) <= tolc + tiny).all()


@pytest.mark.parametrize("precision", [pdgb.PD_PREC_F64, pdgb.PD_PREC_DW])
def test_denormal_seeds(precision):
    # dL/dc = dt/rho s V_j (y/|y|).w of |w| below 1e-309 is zero or a denormal number
    w = workloads.tensile_bar(8, 3, 3, rate=0.0, sc=0.5)
    w.bc_type[:] = 0
    rng = np.random.default_rng(8)
    u0 = 1e-3 * (w.coords - w.coords.mean(0))
    gv = rng.normal(size=(w.n, 3)) * 1e-311
    m = pdgb.Model.from_workload(w, precision=precision)
    m.set_state(u0, np.zeros((w.n, 3)), 0)
    pdgb.pd_adjoint_forward(m.h, 2)
    gc, _, gu0, gv0 = pdgb.pd_adjoint_backward(m.h, np.zeros((w.n, 3)), gv)
    m.close()
    assert (np.abs(gc) < 1e-307).all()
    assert np.isfinite(gu0).all() and np.isfinite(gv0).all()

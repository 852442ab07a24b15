"""The reverse step of double-word handles against the oracle, over equal and unequal volumes,
stiffnesses per bond, rotations, large stretches and scales of the seeds.

Their K d is formed wholly in double-words: 2^-44 of each bond's terms, at most
2 c / L (V_m |w_j| + V_j |w_m|), and the sum of up to 122 terms 2^-47 of them each: 2^-40 of
the majorant in all.  dL/dc = dt/rho s V_j (y/|y|).w: the oracle's s carries 8 2^-53, the
kernel's 2^-44 |eta| / |xi| (from eta . (2 xi + eta)) and 2^-42 of itself (nine operations on
words that are not normalised, 46 bits each, and a condition number of up to 1.5)."""
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


@pytest.mark.parametrize("n_shape", [(5, 4, 3), (13, 7, 6)])
@pytest.mark.parametrize("volumes_vary", [False, True])
@pytest.mark.parametrize("per_bond", [False, True])
@pytest.mark.parametrize("strain,angle", [(1e-5, 0.0), (2e-3, 4e-3), (1e-3, 0.3), (2e-2, 0.0),
                                          (0.1, 1.2), (-0.2, 0.0), (0.6, 0.0)])
@pytest.mark.parametrize("seed_scale", [1.0, 1e-60, 1e50])
def test_reverse_step(n_shape, volumes_vary, per_bond, strain, angle, seed_scale):
    w = workloads.tensile_bar(*n_shape, rate=0.0, sc=5.0)
    rng = np.random.default_rng(9)
    w.bc_type[:] = 0
    if volumes_vary:
        w.coords = w.coords + rng.uniform(-0.2, 0.2, w.coords.shape) * w.dx
        w.volumes = w.volumes * rng.uniform(0.5, 2.0, w.n)
    c, s = np.cos(angle), np.sin(angle)
    A = np.array([[c, -s, 0], [s, c, 0], [0, 0, 1]]) * (1 + strain) - np.eye(3)
    u0 = (w.coords - w.coords.mean(0)) @ A.T + rng.uniform(-0.05, 0.05, (w.n, 3)) * strain * w.dx
    v0 = np.zeros((w.n, 3))
    off, idx = oracle.cut_family(w.coords, w.horizon, w.cuts_array())
    rows = np.repeat(np.arange(w.n), np.diff(off))
    c0 = oracle.micromodulus(w.bulk_modulus, w.horizon)
    cb = np.full(len(idx), c0)
    if per_bond:
        lo, hi = np.minimum(rows, idx), np.maximum(rows, idx)
        cb = c0 * (0.6 + 0.4 * np.sin(1.7 * lo + 0.3 * hi))     # symmetric
        cb = np.abs(cb) + 0.1 * c0
    gu = rng.normal(size=(w.n, 3)) * seed_scale
    gv = rng.normal(size=(w.n, 3)) * 1e-7 * seed_scale
    om = oracle.Model.from_workload(w, off, idx, c=c0, c_bond=cb)
    gc_o, gl_o, gu_o, gv_o = oracle.adjoint(om, 0, 1, u0, v0, om.fresh_bonds(), gu, gv)
    m = pdgb.Model.from_workload(w, precision=pdgb.PD_PREC_DW, c=c0)
    if per_bond:
        m.set_params(c0, w.sc, w.load, w.disp_rate, cb)
    m.set_state(u0, v0, step=0)
    pdgb.pd_adjoint_forward(m.h, 1)
    gc, gl, gu0, gv0 = pdgb.pd_adjoint_backward(m.h, gu, gv)
    m.close()
    xi, eta = w.coords[idx] - w.coords[rows], u0[idx] - u0[rows]
    L = np.linalg.norm(xi, axis=1)
    st = np.abs(np.linalg.norm(xi + eta, axis=1) / L - 1.0)
    e = np.linalg.norm(eta, axis=1) / L
    wa = np.linalg.norm(gv + w.dt * gu, axis=1)
    dr = w.dt / w.density
    tol = dr * np.bincount(rows, 2 * cb / L * (w.volumes[rows] * wa[idx] + w.volumes[idx] * wa[rows]),
                           minlength=w.n)
    assert (np.abs(gu0 - gu_o).max(1) <= 2.0 ** -40 * tol + 4 * 2.0 ** -53 * np.abs(gu).max(1)).all()
    assert np.abs(gv0 - gv_o).max() <= 8 * 2.0 ** -53 * np.abs(gv_o).max()
    tolc = dr * w.volumes[idx] * wa[rows] * (8 * 2.0 ** -53 + 2.0 ** -44 * e + (2.0 ** -42 + 16 * 2.0 ** -53) * st)
    assert (np.abs(gc - gc_o) <= tolc).all()

"""The FP64 and double-word state-based step's double-word bond arithmetic against the
oracle, one step from a given state with v = 0, so that v = dt F / rho.

Both sides form e = |y| - |xi| of a bond with an absolute error of at most 8 2^-53 |xi|
(the oracle, and the literal bonds here) or 2^-44 e.  So the dilation differs by at most
dth = 48 2^-53 + (2^-44 + 300 2^-53) 3 s_max (two sides, the sums of 122 terms and m), and
with |t_ij| <= |xi| ((3 K + 5 G) |theta| + 15 G s) / m_i the force by at most
sum_j V_j |xi| (1/m_i + 1/m_j) ((3 K + 5 G) dth + 15 G 16 2^-53
+ (2^-44 + 300 2^-53) ((3 K + 5 G) 3 + 15 G) s_max)."""
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


@pytest.mark.parametrize("precision", [pdgb.PD_PREC_F64, pdgb.PD_PREC_DW])
@pytest.mark.parametrize("shape,jitter,horizon", [
    ((1, 1, 2), 0.0, 3.01),      # two nodes
    ((8, 4, 1), 0.0, 3.01),      # one slice exactly
    ((11, 3, 1), 0.0, 3.01),     # one slice and a node, odd families
    ((9, 9, 9), 0.25, 3.01),     # unequal volumes, ragged families
    ((12, 11, 10), 0.2, 5.05)])  # families past 256
@pytest.mark.parametrize("strain", [1e-7, 1e-4, 7.7e-3, 7.9e-3, -7.9e-3, 0.2])
@pytest.mark.parametrize("shift,move", [(0.0, 0.0), (-37.3, 60.0)])
def test_one_state_based_step_against_oracle(precision, shape, jitter, horizon, strain, shift, move):
    w = workloads.tensile_bar(*shape, rate=0.0, sc=0.5)
    K = w.bulk_modulus
    G = 0.6 * K if strain > 0 else 0.3 * K
    w.state_based = (K, G)
    w.bc_type[:] = 0
    w.horizon = horizon * w.dx
    rng = np.random.default_rng(3)
    if jitter:
        w.coords = w.coords + rng.uniform(-jitter, jitter, w.coords.shape) * w.dx
        w.volumes = w.volumes * rng.uniform(0.5, 2.0, w.n)
    w.coords = w.coords + shift * w.dx
    A = rng.uniform(-0.3, 0.3, (3, 3)) * strain + np.eye(3) * strain
    u = (w.coords - w.coords.mean(0)) @ A.T + rng.uniform(-0.1, 0.1, (w.n, 3)) * strain * w.dx
    u += move * w.dx
    off, idx = oracle.cut_family(w.coords, w.horizon, w.cuts_array())
    om = oracle.Model.from_workload(w, off, idx)
    uo, vo, mu = u.copy(), np.zeros((w.n, 3)), om.fresh_bonds()
    om.run(0, 1, uo, vo, mu)
    m = pdgb.Model.from_workload(w, precision=precision)
    m.set_state(u, np.zeros((w.n, 3)), 0)
    m.step(1)
    ug, vg = m.state()
    assert np.array_equal(m.bonds(), mu)
    m.close()
    rows = np.repeat(np.arange(w.n), np.diff(off))
    xi = w.coords[idx] - w.coords[rows]
    L = np.linalg.norm(xi, axis=1)
    s_max = np.abs(np.linalg.norm(xi + u[idx] - u[rows], axis=1) / L - 1.0).max()
    mv = np.bincount(rows, L * L * w.volumes[idx], minlength=w.n)
    eps, dw = 2.0 ** -53, 2.0 ** -44 + 300 * 2.0 ** -53
    dth = 48 * eps + dw * 3 * s_max
    per = (3 * K + 5 * G) * dth + 15 * G * 16 * eps + dw * (3 * (3 * K + 5 * G) + 15 * G) * s_max
    tol = np.bincount(rows, w.volumes[idx] * L * (1 / mv[rows] + 1 / mv[idx]), minlength=w.n) * per
    tol = tol * w.dt / w.density + 4 * eps * np.abs(vo).max(1)
    assert (np.abs(vg - vo).max(1) <= tol).all()

"""The FP64 step's double-word bond arithmetic and its split over warps, against the
oracle and against itself.

One step from a given state with v = 0, so that v = dt F / rho: the oracle forms each
bond's stretch literally in FP64, with an absolute error of a few 2^-53 (the roundings
of y, |y|^2, |y| and |xi|), and the kernel has 2^-45 of the force; so the node's
velocity differs by at most dt/rho sum_j c V_j (8 2^-53 + 2^-45 |s_j|) and the rounding
of the sums, 122 2^-53 of their terms."""
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


def _body(shape, jitter, seed, shift, horizon):
    w = workloads.tensile_bar(*shape, rate=0.0, sc=0.5)
    rng = np.random.default_rng(seed)
    w.bc_type[:] = 0
    w.horizon = horizon * w.dx
    if jitter:
        w.coords = w.coords + rng.uniform(-jitter, jitter, w.coords.shape) * w.dx
        w.volumes = w.volumes * rng.uniform(0.5, 2.0, w.n)
    w.coords = w.coords + shift * w.dx
    return w


@pytest.mark.parametrize("shape,jitter,horizon", [
    ((1, 1, 2), 0.0, 3.01),      # two nodes
    ((8, 4, 1), 0.0, 3.01),      # one slice exactly
    ((11, 3, 1), 0.0, 3.01),     # one slice and a node
    ((9, 9, 9), 0.25, 3.01),     # unequal volumes, ragged families
    ((12, 11, 10), 0.2, 5.05),   # families past 256: one warp per slice
    ((40, 10, 10), 0.0, 3.01)])
@pytest.mark.parametrize("strain", [1e-7, 1e-4, 7.7e-3, 7.9e-3, -7.9e-3, 0.2])
@pytest.mark.parametrize("shift,move", [(0.0, 0.0), (1e4, 0.0), (-37.3, 60.0), (0.0, 1e5)])
def test_one_step_against_oracle(shape, jitter, horizon, strain, shift, move):
    w = _body(shape, jitter, 3, shift, horizon)
    rng = np.random.default_rng(7)
    A = rng.uniform(-0.3, 0.3, (3, 3)) * strain + np.eye(3) * strain
    u = (w.coords - w.coords.mean(0)) @ A.T + rng.uniform(-0.1, 0.1, (w.n, 3)) * strain * w.dx
    u += move * w.dx
    off, idx = oracle.cut_family(w.coords, w.horizon, w.cuts_array())
    om = oracle.Model.from_workload(w, off, idx)
    uo, vo, mu = u.copy(), np.zeros((w.n, 3)), om.fresh_bonds()
    om.run(0, 1, uo, vo, mu)
    m = pdgb.Model.from_workload(w, precision=pdgb.PD_PREC_F64)
    m.set_state(u, np.zeros((w.n, 3)), 0)
    m.step(1)
    ug, vg = m.state()
    assert np.array_equal(m.bonds(), mu)
    m.close()
    c = oracle.micromodulus(w.bulk_modulus, w.horizon)
    rows = np.repeat(np.arange(w.n), np.diff(off))
    xi = w.coords[idx] - w.coords[rows]
    L = np.linalg.norm(xi, axis=1)
    s = np.abs(np.linalg.norm(xi + u[idx] - u[rows], axis=1) / L - 1.0)
    # both read u as given, but the oracle's eta is the difference of two rounded sums
    # only through u itself: no further term
    tol = np.zeros(w.n)
    np.add.at(tol, rows, w.volumes[idx] * (8 * 2.0 ** -53 + (2.0 ** -45 + 122 * 2.0 ** -53) * s))
    tol = tol * c * w.dt / w.density + 4 * 2.0 ** -53 * np.abs(vo).max(1)
    assert (np.abs(vg - vo).max(1) <= tol).all()


@pytest.mark.parametrize("shape,jitter", [((6, 6, 5), 0.2), ((40, 10, 10), 0.0),
                                          ((70, 22, 21), 0.1)])
def test_result_does_not_depend_on_the_split(shape, jitter):
    out = []
    for block in (32, 64, 128, 256):   # 1, at most 2, 4 and 8 warps per slice
        w = _body(shape, jitter, 5, 0.0, 3.01)
        w.sc = 1.2e-4                   # some bonds break, some lie near it
        rng = np.random.default_rng(1)
        u = 1e-4 * (w.coords - w.coords.mean(0)) + rng.uniform(-1, 1, (w.n, 3)) * 2e-5 * w.dx
        m = pdgb.Model.from_workload(w, precision=pdgb.PD_PREC_F64, block_threads=block)
        m.set_state(u, np.zeros((w.n, 3)), 0)
        m.step(7)
        out.append((*m.state(), m.bonds(), m.damage()))
        m.close()
    assert 0 < (out[0][2] == 0).sum() < out[0][2].size
    for o in out[1:]:
        for a, b in zip(out[0], o):
            assert np.array_equal(a, b)

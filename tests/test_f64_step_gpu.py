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


@pytest.mark.parametrize("n_shape", [(5, 4, 3), (13, 7, 6)])
@pytest.mark.parametrize("jitter", [0.0, 0.2])       # equal and unequal volumes
@pytest.mark.parametrize("per_bond", [False, True])
@pytest.mark.parametrize("strain,angle", [(1e-5, 0.0), (2e-3, 4e-3), (1e-3, 0.3), (2e-2, 0.0)])
@pytest.mark.parametrize("seed_scale", [1.0, 1e-60, 1e50])
def test_reverse_step_against_oracle(n_shape, jitter, per_bond, strain, angle, seed_scale):
    # one reverse step: dL/du0 = gu + dt/rho sum c K d with w = gv + dt gu, formed by the
    # oracle literally in FP64.  |K d| <= 2 |d| / L and both sides round a dozen
    # operations a bond and the sum: 200 2^-53 of the terms' sum bounds the difference.
    # dL/dc = dt/rho s V_j (y/|y|).w: the oracle's s carries 8 2^-53, the kernel's 2^-44
    # of itself, the other factors a few roundings.
    w = _body(n_shape, jitter, 4, 0.0, 3.01)
    rng = np.random.default_rng(9)
    c, s = np.cos(angle), np.sin(angle)
    A = np.array([[c, -s, 0], [s, c, 0], [0, 0, 1]]) @ (np.eye(3) * (1 + strain)) - np.eye(3)
    u0 = (w.coords - w.coords.mean(0)) @ A.T + rng.uniform(-0.05, 0.05, (w.n, 3)) * strain * w.dx
    v0 = np.zeros((w.n, 3))
    off, idx = oracle.cut_family(w.coords, w.horizon, w.cuts_array())
    c0 = oracle.micromodulus(w.bulk_modulus, w.horizon)
    cb = np.full(len(idx), c0)
    if per_bond:
        cb = workloads.bond_stiffness_grf(w, off, idx, c0, 3)
        rev = workloads.reverse_bond(w.n, off, idx)
        cb = 0.5 * (cb + cb[rev])
    gu = rng.normal(size=(w.n, 3)) * seed_scale
    gv = rng.normal(size=(w.n, 3)) * 1e-7 * seed_scale
    om = oracle.Model.from_workload(w, off, idx, c=c0, c_bond=cb)
    gc_o, gl_o, gu_o, gv_o = oracle.adjoint(om, 0, 1, u0, v0, om.fresh_bonds(), gu, gv)
    m = pdgb.Model.from_workload(w, precision=pdgb.PD_PREC_F64, c=c0)
    if per_bond:
        m.set_params(c0, w.sc, w.load, w.disp_rate, cb)
    m.set_state(u0, v0, step=0)
    pdgb.pd_adjoint_forward(m.h, 1)
    gc, gl, gu0, gv0 = pdgb.pd_adjoint_backward(m.h, gu, gv)
    m.close()
    rows = np.repeat(np.arange(w.n), np.diff(off))
    xi = w.coords[idx] - w.coords[rows]
    L = np.linalg.norm(xi, axis=1)
    s = np.abs(np.linalg.norm(xi + u0[idx] - u0[rows], axis=1) / L - 1.0)
    ww = gv + w.dt * gu
    wa = np.linalg.norm(ww, axis=1)
    dr = w.dt / w.density
    tol = np.zeros(w.n)
    np.add.at(tol, rows, 2 * cb / L * (w.volumes[rows] * wa[idx] + w.volumes[idx] * wa[rows]))
    tol = 200 * 2.0 ** -53 * (dr * tol + np.abs(gu).max(1))
    assert (np.abs(gu0 - gu_o).max(1) <= tol).all()
    assert np.abs(gv0 - gv_o).max() <= 8 * 2.0 ** -53 * np.abs(gv_o).max()
    tolc = dr * w.volumes[idx] * wa[rows] * (8 * 2.0 ** -53 + (2.0 ** -44 + 16 * 2.0 ** -53) * s)
    assert (np.abs(gc - gc_o) <= tolc).all()


def test_handles_that_share_a_kernel_do_not_disturb_each_other():
    # the step's shared memory depends on the model (104 KB a block for families of 256
    # with two warps per slice, 13 KB for the small bar): a handle keeps stepping after one
    # with other needs was made
    big = _body((32, 30, 30), 0.1, 2, 0.0, 3.8)
    small = _body((12, 8, 8), 0.1, 2, 0.0, 3.01)
    out = []
    for between in (False, True):
        m = pdgb.Model.from_workload(big, precision=pdgb.PD_PREC_F64)
        u = 1e-5 * (big.coords - big.coords.mean(0)) ** 2 / big.dx
        m.set_state(u, np.zeros_like(u), 0)
        m.step(2)
        if between:
            k = pdgb.Model.from_workload(small, precision=pdgb.PD_PREC_F64)
            k.step(2)
        m.step(3)
        if between:
            k.step(2)
            assert np.isfinite(k.state()[0]).all()
            k.close()
        out.append(m.state())
        m.close()
    assert np.abs(out[0][0]).max() > 0
    assert np.array_equal(out[0][0], out[1][0]) and np.array_equal(out[0][1], out[1][1])


@pytest.mark.parametrize("jitter", [0.0, 0.2])
@pytest.mark.parametrize("vv", [False, True])
def test_pmb_forms_of_both_precisions_take_the_same_step(jitter, vv):
    # PD_PREC_F64 and PD_PREC_DW without softening, and with kr = 1 (the PMB law), run the
    # same kernel: the same state and bonds bit for bit, bonds that break included; the
    # damage of an intact family is each precision's own rounding of zero
    out = []
    for prec in (pdgb.PD_PREC_F64, pdgb.PD_PREC_DW):
        for kr in (0.0, 1.0):
            w = _body((13, 9, 8), jitter, 6, 0.0, 3.01)
            w.sc, w.kr = 1.2e-4, kr
            rng = np.random.default_rng(2)
            u = 1e-4 * (w.coords - w.coords.mean(0)) + rng.uniform(-1, 1, (w.n, 3)) * 2e-5 * w.dx
            kw = dict(integrator=pdgb.PD_INTEGRATOR_VV) if vv else {}
            m = pdgb.Model.from_workload(w, precision=prec, **kw)
            m.set_state(u, np.zeros((w.n, 3)), 0)
            m.step(6)
            out.append((*m.state(), m.bonds(), m.damage()))
            m.close()
    assert 0 < (out[0][2] == 0).sum() < out[0][2].size
    for o in out[1:]:
        for a, b in zip(out[0][:3], o[:3]):
            assert np.array_equal(a, b)
    assert np.array_equal(out[0][3], out[1][3]) and np.array_equal(out[2][3], out[3][3])
    assert np.abs(out[0][3] - out[2][3]).max() <= 1e-12

"""The reverse step of FP64 handles over the whole range of stretches of its double-word part.

One reverse step, dL/du0 = gu + dt/rho sum c K d with w = gv + dt gu, against the oracle's
literal FP64.  |K d| <= 2 |d| / L and both sides round a dozen operations a bond and the sum:
200 2^-53 of the terms' sum bounds the difference.  The double-word part has 2^-44 of
|s| |K d|, at most 2^-51 of it here, 4 2^-53 more."""
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


@pytest.mark.parametrize("strain", [1e-3, 3e-3, 5e-3, 6.5e-3, 7.6e-3, -3e-3, -6.5e-3, -7.6e-3])
@pytest.mark.parametrize("volumes_vary", [False, True])
def test_reverse_step(strain, volumes_vary):
    w = workloads.tensile_bar(9, 5, 4, rate=0.0, sc=0.5)
    rng = np.random.default_rng(3)
    w.bc_type[:] = 0
    if volumes_vary:
        w.coords = w.coords + rng.uniform(-0.2, 0.2, w.coords.shape) * w.dx
        w.volumes = w.volumes * rng.uniform(0.5, 2.0, w.n)
    u0 = (w.coords - w.coords.mean(0)) * strain
    v0 = np.zeros((w.n, 3))
    off, idx = oracle.cut_family(w.coords, w.horizon, w.cuts_array())
    c = oracle.micromodulus(w.bulk_modulus, w.horizon)
    gu, gv = np.zeros((w.n, 3)), rng.normal(size=(w.n, 3))
    om = oracle.Model.from_workload(w, off, idx, c=c)
    _, _, gu_o, _ = oracle.adjoint(om, 0, 1, u0, v0, om.fresh_bonds(), gu, gv)
    m = pdgb.Model.from_workload(w, precision=pdgb.PD_PREC_F64, c=c)
    m.set_state(u0, v0, step=0)
    pdgb.pd_adjoint_forward(m.h, 1)
    _, _, gu0, _ = pdgb.pd_adjoint_backward(m.h, gu, gv)
    m.close()
    rows = np.repeat(np.arange(w.n), np.diff(off))
    L = np.linalg.norm(w.coords[idx] - w.coords[rows], axis=1)
    wa = np.linalg.norm(gv, axis=1)
    tol = np.bincount(rows, 2 * c / L * (w.volumes[rows] * wa[idx] + w.volumes[idx] * wa[rows]),
                      minlength=w.n)
    assert (np.abs(gu0 - gu_o).max(1) <= 204 * 2.0 ** -53 * w.dt / w.density * tol).all()

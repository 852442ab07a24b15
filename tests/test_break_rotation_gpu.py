"""Break decisions in a rotated body, on the handles of the three-word step: every bond of a
line of nodes that is stretched evenly by e and turned has s = e to 1e-10 of itself (the
rounding of u), so an s_c that differs by more decides all of them."""
import numpy as np
import pytest

import paper_2105_04150_gb300 as pdgb
import workloads

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _need_gpu():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    pdgb.build()


@pytest.mark.parametrize("precision", [pdgb.PD_PREC_F64, pdgb.PD_PREC_DW])
@pytest.mark.parametrize("state_based", [False, True])
@pytest.mark.parametrize("angle", [0.0, 0.003, 0.01, 0.1, 1.2])
@pytest.mark.parametrize("off", [1e-8, 1e-6, 1e-5, 1e-4, 1e-2])
@pytest.mark.parametrize("e", [1e-5, 1e-4, 3e-3])
def test_decisions(precision, state_based, angle, off, e):
    for sign in (-1, 1):
        w = workloads.tensile_bar(40, 1, 1, rate=0.0, sc=e * (1 + sign * off))
        w.bc_type[:] = 0
        if state_based:
            w.state_based = (w.bulk_modulus, 0.6 * w.bulk_modulus)
        c, s = np.cos(angle), np.sin(angle)
        d = np.array([c, 0.6 * s, 0.8 * s])
        x = w.coords[:, 0] - w.coords[:, 0].mean()
        u = (1 + e) * x[:, None] * d - x[:, None] * np.array([1.0, 0.0, 0.0])
        m = pdgb.Model.from_workload(w, precision=precision)
        m.set_state(u, np.zeros((w.n, 3)), 0)
        m.step(1)
        mu = m.bonds()
        m.close()
        assert (mu == (0 if sign < 0 else 1)).all()


@pytest.mark.parametrize("precision", [pdgb.PD_PREC_F64, pdgb.PD_PREC_DW])
@pytest.mark.parametrize("angle", [0.0, 0.01, 0.1, 1.2])
@pytest.mark.parametrize("off", [1e-6, 1e-5, 1e-4, 1e-2])
def test_decisions_of_the_softening_step(precision, angle, off):
    # kr = 1 with no-fail nodes runs the softening kernels; s_0 = s_c.  The double-word one
    # forms s itself, from u to 2^-48 of it (20 spacings here): 1e-12, 1e-8 of s_c
    e = 1e-4
    for sign in (-1, 1):
        w = workloads.tensile_bar(40, 1, 1, rate=0.0, sc=e * (1 + sign * off))
        w.bc_type[:] = 0
        w.kr = 1.0
        w.no_fail = (np.arange(w.n) >= 35).astype(np.uint8)
        c, s = np.cos(angle), np.sin(angle)
        d = np.array([c, 0.6 * s, 0.8 * s])
        x = w.coords[:, 0] - w.coords[:, 0].mean()
        u = (1 + e) * x[:, None] * d - x[:, None] * np.array([1.0, 0.0, 0.0])
        m = pdgb.Model.from_workload(w, precision=precision)
        off_, idx = m.family()
        rows = np.repeat(np.arange(w.n), np.diff(off_))
        m.set_state(u, np.zeros((w.n, 3)), 0)
        m.step(1)
        mu = m.bonds()
        m.close()
        can = (rows < 35) & (idx < 35)
        assert (mu[~can] == 1).all()
        assert (mu[can] == (0 if sign < 0 else 1)).all()

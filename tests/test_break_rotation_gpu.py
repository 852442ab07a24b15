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

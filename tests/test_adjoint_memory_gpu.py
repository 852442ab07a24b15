"""Device memory of the reverse sweep: what the header states, every buffer rounded up to at
least 256 bytes, and nothing more on later calls."""
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
def test_device_memory_of_the_reverse_sweep(precision):
    w = workloads.tensile_bar(40, 10, 10, rate=0.0, sc=0.5)
    m = pdgb.Model.from_workload(w, precision=precision)
    pdgb.pd_adjoint_forward(m.h, 4)
    held = [m.info()["device_bytes"]]
    g = np.ones((w.n, 3))
    for want_c in (False, True, True):
        pdgb.pd_adjoint_backward(m.h, g, want_c=want_c)
        held.append(m.info()["device_bytes"])
    info = m.info()
    m.close()
    pad = (w.n + 31) // 32 * 32
    slots = pad * info["ell_width"]
    per_slot = 32 if precision == pdgb.PD_PREC_F64 else 8
    assert 0 < held[1] - held[0] - (384 * pad + per_slot * slots) <= 16 * 256
    assert 0 <= held[2] - held[1] - (8 * w.n + 12 * info["n_bonds"]) <= 256
    assert held[3] == held[2]

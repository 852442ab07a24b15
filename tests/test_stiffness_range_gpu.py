"""Stiffnesses per bond outside FP32's range (18 K / (pi delta^4) passes 3.4e38 at horizons
below 0.2 um in SI units).

With every stiffness, the density and the damping multiplied by the same power of two the
accelerations are the same numbers, and so are u, v and the gradients; dL/dc is divided by
that power.  Nothing rounds differently: the comparison is exact."""
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


def _run(precision, power, jitter, strain):
    f = 2.0 ** power
    w = workloads.tensile_bar(9, 6, 5, rate=0.0, sc=0.5)
    rng = np.random.default_rng(6)
    w.bc_type[:] = 0
    w.density, w.damping = w.density * f, w.damping * f
    if jitter:
        w.coords = w.coords + rng.uniform(-jitter, jitter, w.coords.shape) * w.dx
        w.volumes = w.volumes * rng.uniform(0.5, 2.0, w.n)
    off, idx = oracle.cut_family(w.coords, w.horizon, w.cuts_array())
    c0 = oracle.micromodulus(w.bulk_modulus, w.horizon)
    cb = c0 * rng.uniform(0.5, 2.0, len(idx))
    x = w.coords - w.coords.mean(0)
    u0 = strain * x + rng.uniform(-0.1, 0.1, (w.n, 3)) * strain * w.dx
    m = pdgb.Model.from_workload(w, precision=precision, c=c0)
    m.set_params(c0 * f, w.sc, w.load, w.disp_rate, cb * f)
    m.set_state(u0, np.zeros((w.n, 3)), 0)
    m.step(5)
    out = list(m.state())
    m.set_state(u0, np.zeros((w.n, 3)), 0)
    pdgb.pd_adjoint_forward(m.h, 4)
    gc, _, gu, gv = pdgb.pd_adjoint_backward(m.h, rng.normal(size=(w.n, 3)),
                                             rng.normal(size=(w.n, 3)) * 1e-6)
    m.close()
    return out + [gc * f, gu, gv]


@pytest.mark.parametrize("precision", [pdgb.PD_PREC_F64, pdgb.PD_PREC_DW])
@pytest.mark.parametrize("jitter", [0.0, 0.2])
@pytest.mark.parametrize("strain", [1e-4, 2e-2])       # double-words; mostly literal
def test_scaled_stiffness_gives_the_same_run(precision, jitter, strain):
    ref = _run(precision, 0, jitter, strain)
    assert all(np.isfinite(a).all() and np.abs(a).max() > 0 for a in ref)
    for power in (100, -230):
        for a, b in zip(ref, _run(precision, power, jitter, strain)):
            assert np.array_equal(a, b)

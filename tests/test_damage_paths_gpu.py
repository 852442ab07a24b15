"""The damage is a function of the bond flags: what a step writes and what pd_damage forms by
itself (after the bonds were set, or after a gradient call that leaves the state as it was)
are the same numbers, bit for bit, on the handles that run the three-word step."""
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
@pytest.mark.parametrize("jitter", [0.0, 0.2])       # equal and unequal volumes
@pytest.mark.parametrize("state_based", [False, True])
@pytest.mark.parametrize("broken", [False, True])
def test_damage_of_the_same_flags(precision, jitter, state_based, broken):
    w = workloads.tensile_bar(13, 9, 8, rate=0.0, sc=1.2e-4 if broken else 0.5)
    rng = np.random.default_rng(2)
    w.bc_type[:] = 0
    if state_based:
        w.state_based = (w.bulk_modulus, 0.6 * w.bulk_modulus)
    if jitter:
        w.coords = w.coords + rng.uniform(-jitter, jitter, w.coords.shape) * w.dx
        w.volumes = w.volumes * rng.uniform(0.5, 2.0, w.n)
    u = 1e-4 * (w.coords - w.coords.mean(0)) + rng.uniform(-1, 1, (w.n, 3)) * 2e-5 * w.dx
    m = pdgb.Model.from_workload(w, precision=precision)
    m.set_state(u, np.zeros((w.n, 3)), 0)
    m.step(3)
    mu, after_step = m.bonds(), m.damage()
    assert (mu == 0).any() == broken
    m.set_bonds(mu)
    assert np.array_equal(m.damage(), after_step)
    m.set_state(*m.state(), 3)
    assert np.array_equal(m.damage(), after_step)
    if not state_based:
        m.step(1)
        mu, after_step = m.bonds(), m.damage()
        pdgb.pd_adjoint_forward(m.h, 2)
        pdgb.pd_adjoint_backward(m.h, np.ones((w.n, 3)))
        assert np.array_equal(m.bonds(), mu)
        assert np.array_equal(m.damage(), after_step)
    m.close()

"""dL/dc of a long recorded run is the sum of one term a step for every bond.

The terms come from the same kernels, one reverse step at a time: each step is recorded
and swept by itself with the gradient that the step after it left, so they are the terms
of the long sweep bit for bit (the scale of the double-words is a power of two).  Their
sum in long double is compared with the long sweep's dL/dc.

The sum is an FP64 one, one rounding of at most 2^-53 of the running sum a step, and the
result is scaled by dt/rho V and 1/scale (each single term too): (N + 8) 2^-53 sum |g_k|."""
import numpy as np
import pytest

import oracle
import paper_2105_04150_gb300 as pdgb
import workloads

pytestmark = pytest.mark.gpu

N = 1500


@pytest.fixture(scope="module", autouse=True)
def _need_gpu():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    pdgb.build()


@pytest.mark.parametrize("jitter", [0.0, 0.2])
@pytest.mark.parametrize("precision", [pdgb.PD_PREC_F64, pdgb.PD_PREC_DW])
def test_stiffness_gradient_is_the_sum_of_its_steps(precision, jitter):
    w = workloads.tensile_bar(5, 4, 3, rate=0.0, sc=0.5)
    rng = np.random.default_rng(4)
    w.bc_type[:] = 0
    w.dt = 2e-9        # slow against the waves: terms of one sign add up
    if jitter:
        w.coords = w.coords + rng.uniform(-jitter, jitter, w.coords.shape) * w.dx
        w.volumes = w.volumes * rng.uniform(0.5, 2.0, w.n)
    u0 = 1e-3 * (w.coords - w.coords.mean(0)) + rng.uniform(-1, 1, (w.n, 3)) * 1e-4 * w.dx
    gu, gv = rng.normal(size=(w.n, 3)), rng.normal(size=(w.n, 3)) * 1e-6
    m = pdgb.Model.from_workload(w, precision=precision)
    m.set_state(u0, np.zeros((w.n, 3)), 0)
    states = []
    for k in range(N):
        states.append(m.state())
        m.step(1)
    total = abs_total = 0
    du, dv = gu, gv
    for k in reversed(range(N)):
        m.set_state(*states[k], k)
        pdgb.pd_adjoint_forward(m.h, 1)
        g, _, du, dv = pdgb.pd_adjoint_backward(m.h, du, dv)
        total = total + g.astype(np.longdouble)
        abs_total = abs_total + np.abs(g)
    m.set_state(u0, np.zeros((w.n, 3)), 0)
    pdgb.pd_adjoint_forward(m.h, N)
    g, _, du1, dv1 = pdgb.pd_adjoint_backward(m.h, gu, gv)
    m.close()
    assert np.array_equal(du, du1) and np.array_equal(dv, dv1)
    assert (abs_total > 0).all()
    rel = np.abs(np.asarray(g - total, np.float64)) / abs_total
    assert rel.max() <= (N + 8) * 2.0 ** -53

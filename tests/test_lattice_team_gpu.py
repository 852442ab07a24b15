"""The FP32 lattice step with four warps per slice against the one with one warp per slice:
the same operations in the same order per node, so the same bits."""
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


@pytest.mark.parametrize("shape", [
    (8, 2, 2),      # one slice exactly
    (11, 3, 2),     # two slices and two nodes
    (38, 24, 16),   # 456 slices, the largest that take four warps
    (457, 8, 4),    # 457 slices
    (29, 20, 25)])  # 453.1 slices
@pytest.mark.parametrize("hashed", [False, True])
@pytest.mark.parametrize("strain", [5e-5, 6e-3])   # bonds near s_c; past the series too
def test_four_warps_per_slice_equal_one_bitwise(shape, hashed, strain):
    w = workloads.tensile_bar(*shape, rate=1e-7, slab=1)
    w.sc = 1e-4
    if hashed:
        w.sc_hash = (7, 9e-5, 1.1e-4)
    w.no_fail = (w.coords[:, 0] < np.median(w.coords[:, 0])).astype(np.uint8)
    rng = np.random.default_rng(3)
    u = strain * (w.coords - w.coords.mean(0))
    u = u + rng.uniform(-1, 1, u.shape) * 4e-5 * w.dx
    out = []
    for variant in (0, 1):
        m = pdgb.Model.from_workload(w, precision=pdgb.PD_PREC_F32, lat_variant=variant)
        assert m.info()["lat_variant"] == variant
        m.set_state(u, np.zeros_like(u), 0)
        m.step(9)
        out.append((*m.state(), m.bonds(), m.damage()))
        m.close()
    assert (out[0][2] == 0).any() and (out[0][2] == 1).any()
    for a, b in zip(*out):
        assert np.array_equal(a, b)

"""The bench's step footprint (its evidence that a step's arrays exceed the L2) per model."""
import pytest

import bench

N, B = 1000, 122000


@pytest.mark.parametrize("precision,osb,kr,per_bond,per_node", [
    (32, False, 0.0, 4.125, 93),
    (32, True, 0.0, 4.125, 93 + 16),
    (32, False, 2.0, 4.125 + 4, 93),
    # the three-word step: U / |xi| 8 B a slot; two 64-byte records, u 64, v 48, 21 more
    (64, False, 0.0, 12.125, 261), (48, False, 0.0, 12.125, 261),
    (64, False, 1.0, 12.125, 261), (48, False, 1.0, 12.125, 261),
    (64, True, 0.0, 12.125, 261 + 40), (48, True, 0.0, 12.125, 261 + 40),
    # softening: 1/|xi| or |xi| 8 B and the integrity 8 B a slot
    (64, False, 2.0, 20.125, 193), (48, False, 2.0, 20.125, 305)])
def test_step_footprint(precision, osb, kr, per_bond, per_node):
    got = bench.step_footprint(N, B, precision, False, osb, kr)
    assert got == B * per_bond + N * per_node
    assert bench.model_bytes(precision, osb, kr) == (per_bond, per_node)

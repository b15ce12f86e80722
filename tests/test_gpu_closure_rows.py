"""The closure step on rows that are not whole 128-cell tiles.

The tiles of the fused network then run on across the padded rows of a plane.
The same two comparisons as for rows of whole tiles, at their tolerance: against
the reference at the kernels' precision, and a zero network and a dead zone
wider than every prediction against plain updates bit for bit. Rows that fill
their padding (62 of 64 positions) and that just miss it (63 of 72), odd
extents, planes of less than a tile and of a tile and a bit, blocks with one
tile and with several, and (9, 8, 7), which the separate network still takes.
"""
import pytest

import test_gpu_closure as T

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [
    (24, 20, 18), (15, 14, 13), (14, 9, 40), (62, 30, 20), (63, 18, 16), (130, 14, 12),
    (250, 40, 17), (9, 8, 7),
])
def test_closure_step(shape):
    T.test_closure_step_matches_oracle_and_zero_network_is_rr(shape)


@pytest.mark.parametrize("shape", [(24, 20, 18), (65, 17, 16)])
def test_closure_step_with_a_dead_zone(shape):
    T.test_closure_step_with_a_dead_zone_matches_oracle(shape)

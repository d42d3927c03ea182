"""Host-side arithmetic of the workspace layout (runs without a GPU)."""
import pytest


# the fixed array of the allocation-free entry is checked against the end of the forward arrays alone: everything that forming
# log-probabilities touches has to lie before it, also from 32769 rows on, where the mask scan is a pass of its own
@pytest.mark.parametrize("static_scratch", [False, True])
@pytest.mark.parametrize("T", [1, 32768, 32769, 40000, 262145, 2 ** 21])
@pytest.mark.parametrize("d,V", [(64, 300), (64, 32768), (2048, 151936)])
def test_forward_arrays_end_where_the_slab_starts(T, d, V, static_scratch):
    from paper_2512_21450_b200.binding import debug_workspace
    total, forward, row_pos_end = debug_workspace(T, d, V, static_scratch=static_scratch)
    assert 0 < row_pos_end <= forward <= total
    assert forward >= T * (2 * d + 28 + 16 * 16) + (4 * T if T > 32768 else 0)

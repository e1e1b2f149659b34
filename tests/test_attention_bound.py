"""The error bound of the attention kernel's test by entries, on the CPU: it has room for hi and lo planes of both operands and none for
a kernel that lost one of them."""
import pytest

from tests.test_attention_gpu import TILE_CASES, definition_and_bound, tile_case


@pytest.mark.parametrize("case", TILE_CASES)
def test_bound_notices_a_lost_plane(case):
    q, kv, pos = tile_case(*case)
    args = (q, kv, pos, case[1], sorted({0, case[0] - 1}))
    ref, bound = definition_and_bound(*args)

    def worst(q_lo, p_lo):
        return ((definition_and_bound(*args, q_lo=q_lo, p_lo=p_lo)[0] - ref).abs() / bound).max().item()
    assert worst(True, True) < 0.2
    assert worst(False, True) > 1.5
    assert worst(True, False) > 1.5

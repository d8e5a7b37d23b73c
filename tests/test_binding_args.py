"""Argument marshalling of the binding (no device needed)."""
import ctypes

import pytest


def arrays(sd):
    n = sd.c.batch
    get = lambda at, k: list((ctypes.c_int32 * k).from_address(at))
    return get(sd.c.row_off, n + 1), get(sd.c.rank, n), get(sd.c.rank_off, n + 1)


def test_sequence_arrays():
    from paper_2403_02352_b200.binding import SeqDesc
    sd = SeqDesc([5, 0, 7], [2, 0, 3])
    assert arrays(sd) == ([0, 5, 5, 12], [2, 0, 3], [0, 2, 2, 5])
    assert (sd.total_rows, sd.total_rank) == (12, 5)
    assert arrays(SeqDesc([], [])) == ([0], [], [0])


@pytest.mark.parametrize("lengths,ranks", [([8], [2 ** 32 + 3]), ([8], [2 ** 31]), ([2 ** 32 + 8], [3]), ([2 ** 30, 2 ** 30], [1, 1])])
def test_what_32_bits_do_not_hold_is_refused(lengths, ranks):
    from paper_2403_02352_b200.binding import SeqDesc
    with pytest.raises(OverflowError):
        SeqDesc(lengths, ranks)

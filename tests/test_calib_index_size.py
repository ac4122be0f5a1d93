"""svt_calib_index_size: callers keep the size they once asked for, so the index
of no track set may grow (no GPU needed: the size is plain arithmetic)."""
import pytest


def kept_size(n, S):
    """Counts of 1024-track tiles, the sectors' offsets and first items, the
    items' sectors and first tracks, and their number, at multiples of 256 bytes."""
    items = -(-n // 256) + S
    return sum(-(-4 * k // 256) * 256 for k in (S * -(-n // 1024) + 1, S + 1, S + 1, items, items, 1))


@pytest.mark.parametrize("S", [1, 2, 16, 63, 64, 337, 512])
def test_the_index_does_not_outgrow_earlier_buffers(S):
    from paper_1311_0380_gb300 import _native as N
    L = N.load()
    for n in [0, 1, 31, 1000, 1024, 1025, 2047, 2048, 2049, 3073, 4096, 4097, 64_432, 1_000_003,
              16_000_003, (1 << 31) - 1]:
        assert L.svt_calib_index_size(n, S) <= kept_size(n, S), n

"""Device memory of the ball's table of reads."""
import pytest


@pytest.mark.parametrize("P", [50, 200, 500])
def test_read_table_is_no_larger_than_a_square_of_16_byte_chords(P):
    """Two radii of one lattice differ by their row prefixes (2 pairs of 16 bytes per row and unit of
    radius) and their tables; buffers start at multiples of 256 bytes."""
    from paper_2410_19075_gb300 import workspace_bytes
    N1, P0 = 1001, 8  # no x-window arrays from P = 8 on (8 GiB)
    extra = workspace_bytes(0, 2, N1, P) - workspace_bytes(0, 2, N1, P0) - 2 * 16 * (P - P0) * N1 ** 2
    assert 0 < extra < 16 * (2 * P + 1) ** 2 + 512

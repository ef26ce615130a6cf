"""The bench's count of the several-right-hand-side far field's flops: symmetric
launches carry half of the part that both directions of a pair share, and one
vector in a symmetric launch costs what the headline counts per pair."""
import bench


def test_symmetric_launches_count_the_shared_part_once():
    pairs = 1000
    one_sided = bench.multi_flops(1, 0, 8, pairs)
    assert abs(one_sided - (80.5 + 8 * 8.7) * pairs) < 1e-6 * one_sided
    assert abs(bench.multi_flops(1, 1, 1, pairs) - bench.FLOPS_PER_PAIR * pairs) < 0.1 * pairs
    mixed = bench.multi_flops(3, 2, 14, pairs)  # launches of 8, 5 and 1 vectors
    assert abs(mixed - (one_sided + bench.multi_flops(1, 1, 5, pairs) + bench.multi_flops(1, 1, 1, pairs))) < 1e-6 * mixed

"""The operation and byte counts behind bench.py's roofline figures."""


def test_operations_and_bytes_follow_the_draws_and_the_state():
    """A Gaussian RB linear site that moves back draws nothing, and its state is 20 bytes."""
    import bench
    assert bench.ops_per_site_update({0: 1.0}, 0.02) == 14 + 103 * 0.02
    c3 = bench.ops_per_site_update({3: 1.0}, 0.18)
    assert abs(c3 - (14 + 103 * 0.27 * 0.18)) < 1e-12 and c3 < 20
    assert bench.STATE_BYTES == {0: 4 + 4 + 8, 1: 4 + 4 + 8 + 4 + 8 + 4, 2: 4 + 4, 3: 4 + 4 + 8 + 4, 4: 4 + 4 + 8 + 4 + 8 + 4}

"""Algorithmic bytes with byte sums: one byte less per node written than with 16-bit sums."""
import bench


def test_byte_sums_write_one_byte_per_node():
    a1, nodes = bench.algorithmic_bytes(sum_bytes=1)
    a2, _ = bench.algorithmic_bytes()
    px = sum(w * h for (w, h, _, _) in bench.level_geometry())
    assert a1["aggregate"] == 2 * (2 * nodes + 2 * px)
    assert a2["aggregate"] - a1["aggregate"] == 2 * nodes      # both views
    assert a1["wta"] == a2["wta"] and a1["cost"] == a2["cost"]
    m1, _ = bench.algorithmic_bytes(variant="paper", sum_bytes=1)
    m2, _ = bench.algorithmic_bytes(variant="paper")
    assert m1 == m2                                            # the layers store 16 bits

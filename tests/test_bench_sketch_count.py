"""The bench's sketch roofline counts products, not launches."""
import pytest

import bench


def test_averages_are_per_sketch():
    f, b = bench.sketch_work(20000, 10000, [60] * 5, pure=True, esz=4)
    r = bench.sketch_roofline(f, b, 2.75, 10, "TF32", None, 5)      # each product and the addition of its pieces
    assert r["launches"] == 10 and r["sketches"] == 5
    assert r["avg_ms"] == pytest.approx(0.55)
    assert r["algorithmic_bytes_per_launch"] == pytest.approx(b / 5) and r["algorithmic_flops_per_launch"] == pytest.approx(f / 5)

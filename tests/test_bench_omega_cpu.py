"""The bench's line for omega with the Gram in its kernel (host arithmetic
only): the MMAs as issued for rows in full, of the path the library says it
took, and none for rows as lists."""
import os
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.mark.parametrize("d,tiles_full", [(64, 1000), (70, 1000), (1558, 0)])
def test_rows_in_full(d, tiles_full):
    """Also where the tree took no sweep (a small set's stored distances): its omega issues MMAs all the same."""
    sys.path.insert(0, ROOT)
    import bench
    prof = [{"omega_gram_blocks": 1000, "omega_gram_direct_pairs": 5000, "mst_tiles_full": tiles_full,
             "omega_path": "gram_tc"}]
    r = bench.omega_fused_roofline(prof, {"bf16_tflops": 1900.0}, "measured", 40.0, 152, 2.0, 1900, d, 1e11)
    tensor = r if r["bound"] == "tensor" else r["other_unit"]
    vector = r["other_unit"] if r["bound"] == "tensor" else r
    d_pad = -(-d // 16) * 16
    assert tensor["achieved"] == pytest.approx(1000 * 34 * 2 * 128 * 64 * d_pad / 2e-3 / 1e12)
    assert vector["achieved"] == pytest.approx((1900 * 4096 * 147 + 5000 * (18.75 * d + 95)) / 2e-3 / 1e12)
    assert "tcgen05" in r["kernel"]


def test_rows_as_lists():
    sys.path.insert(0, ROOT)
    import bench
    prof = [{"omega_gram_blocks": 1000, "omega_gram_direct_pairs": 0, "mst_tiles_full": 0, "omega_path": "gram_lists"}]
    r = bench.omega_fused_roofline(prof, {"bf16_tflops": 1900.0}, "measured", 40.0, 152, 2.0, 1900, 4096, 1e11)
    assert r["bound"] == "alu" and r["other_unit"]["achieved"] == 0.0 and "lists" in r["kernel"]

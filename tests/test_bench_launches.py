"""The number of kernels that bench.py reports for a prefill, by hand."""
import bench


def test_prefill_launches():
    assert bench._prefill_launches(289, 12, 152) == 2 + 1 + 12 * 7 + 1
    assert bench._prefill_launches(96 * 152, 2, 152) == 2 + 1 + 2 * 7 + 1
    assert bench._prefill_launches(96 * 152 + 1, 2, 152) == 2 + 2 * (1 + 2 * 7 + 1)

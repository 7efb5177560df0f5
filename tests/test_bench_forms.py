"""bench.py charges the FP64 instruction counts by the forms that ran (host only)."""
import bench


def test_products_share():
    assert bench.products_share([30, 0, 0, 0]) == 1.0
    assert bench.products_share([0, 0, 30, 0]) == 0.0
    assert bench.products_share([10, 0, 30, 0]) == 0.25
    for forms in ([0, 0, 0, 0], [0, 30, 0, 0], [29, 0, 0, 1], [0, 0, 29, 1]):
        assert bench.products_share(forms) is None

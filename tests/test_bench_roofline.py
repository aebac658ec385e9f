"""The tensor-core roofline counts the digit pairs of the path it describes: 15
per real product in mixed precision, 36 in FP64."""
import pytest


@pytest.mark.parametrize("mixed,pairs", [(True, 15), (False, 36)])
def test_tensor_core_roofline(mixed, pairs):
    import bench
    r = bench.tc_roofline({"tc": {"ms": 1000.0, "flops": 4e12}}, {"bf16_tflops_sustained": 1754.4}, mixed)
    assert r["achieved"] == 4.0
    assert r["bf16_tflops_achieved"] == pytest.approx(4.0 * 3 * pairs / 4)
    assert r["frac"] == pytest.approx(4.0 * 3 * pairs / 4 / 1754.4)

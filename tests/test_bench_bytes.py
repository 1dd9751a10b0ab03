"""The bytes the benchmark says a kernel moves at least.  Where an instance
stays on chip for all n updates, f crosses DRAM once per launch, so the figure
is below the two-pass kernels' (which cross it in every update) however many
updates the launch has.  No GPU needed."""
import pytest


@pytest.mark.parametrize("precision,f_value,ref", [("fp32", 4, 4), ("fp16s", 2, 4), ("bf16s", 2, 4)])
def test_onchip_bytes_are_per_launch(precision, f_value, ref):
    import bench
    f = 2 * 19 * f_value  # two components, 19 directions
    coordinates_and_word, fields = 8, 5 * 4
    want = 2 * f + 2 * ref + coordinates_and_word + fields
    assert bench.alg_bytes_per_cell("onchip", precision) == want
    assert want / 2 < bench.alg_bytes_per_cell("persistent", precision)  # two updates already

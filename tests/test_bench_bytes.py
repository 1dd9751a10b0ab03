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


def test_captured_figures_are_of_these_sources():
    """The DRAM traffic and the FP64 operation count were captured from the kernels as they
    are; a change of their code needs new captures, or the benchmark's line loses `traffic`,
    the wasted-traffic ratio and, in FP64, the bound of the FP64 pipe."""
    import bench
    for entry in (bench.NCU_TRAFFIC["k_collide_c2/fp16s/spheres"], bench.FP64_FLOPS["k_collide_c"]):
        assert entry["src"] == bench.sources_hash(entry["files"])


def test_comments_do_not_void_captured_figures():
    import bench
    code = "int a = 1;\nint b = a / 2;\n"
    assert bench.code_only("// one\nint a = 1; /* two\n three */\n\n  int b = a / 2;  // four\n") == bench.code_only(code)
    assert bench.code_only(code.replace("2", "3")) != bench.code_only(code)

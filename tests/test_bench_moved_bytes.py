"""The bytes that the bench's roofline fields count, from the kernels' arrays (no GPU)."""
import bench


def test_moved_bytes_are_those_of_the_arrays():
    F, real, record = 19 * 4, 4, 4 * 4  # FP32: populations, phi, colour or gradient record
    assert bench.moved_bytes_per_node("phi", "fp32") == F + record + real
    assert bench.moved_bytes_per_node("grad_wetting", "fp32") == real + record
    assert bench.moved_bytes_per_node("collide", "fp32") == F + real + record + F + record == 188
    assert bench.moved_bytes_per_node("collide", "fp16") == 38 * 2 + real + 2 * record == 112
    # a step of the bench's line counts these three kernels
    assert sum(bench.moved_bytes_per_node(k, "fp32") for k in ("phi", "grad_wetting", "collide")) == 304

"""The step kernel that a benchmark line names is the one that the lattice runs on."""
import os
import sys

sys.path.insert(0, os.path.dirname(os.path.dirname(os.path.abspath(__file__))))


def test_kernel_names():
    import bench
    m1, e5, other = [5, 12, 14, 17, 21, 26], [1, 14, 49, 51, 60, 70], [1, 2, 3, 6, 7, 11]
    assert bench.kernel_name("f64", 0, m1, 65536, 152) == "fused_f64_kernel<StencilDef<5,12,14,17,21,26>>"
    assert bench.kernel_name("f64", 0, e5, 65536, 152) == "fused_f64_kernel<StencilDef<1,14,49,51,60,70>>"
    assert bench.kernel_name("f64", 0, other, 65536, 152) == "step_f64_kernel"
    assert bench.kernel_name("f64", 0, other, 4864, 152) == "lanes64_kernel"
    assert bench.kernel_name("f32", 3, e5, 100) == "fused_f32_kernel<StencilDef<1,14,49,51,60,70>, false>"
    assert bench.kernel_name("f32", 0, other, 100) == "step_f32_kernel<64>"

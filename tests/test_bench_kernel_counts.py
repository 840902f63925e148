"""The benchmark's counts for the kernels that run, by hand from their operand
layouts: the row-marching kernels (staging "auto") and the per-tile ones, and the
source files that a recorded DRAM traffic belongs to."""
import pytest

from paper_2609_09020_gb300 import workloads as wk


@pytest.fixture(scope="module")
def bench():
    import bench as b
    return b


def _workload(net, L, C, act="relu"):
    return wk.custom("count", 64, 64, L, C, net, act=act, weight_dtype="fp16", precisions=("fp16_tc",))


def test_tensor_macs_of_the_marching_kernels(bench):
    macs = bench.march_tensor_macs_per_px
    # 7-64-64-3: 4 pairs of features, hi and lo, the bias in the odd one's place: K = 16;
    # hidden K = 64 + 64 and a bias step; output layer N = 16, its bias added in fp32
    assert macs(wk.WORKLOADS["c5"]) == 16 * 64 + (128 + 16) * 64 + 128 * 16
    # 14-64-64-3: 7 pairs twice and the bias column in K = 32
    assert macs(wk.WORKLOADS["c3"]) == 32 * 64 + (128 + 16) * 64 + 128 * 16
    # 16-64-64-64-3: 8 pairs twice fill K = 32, so layer 0 has a bias step; output layer in fp32
    assert macs(wk.WORKLOADS["c4"]) == (32 + 16) * 64 + 2 * (128 + 16) * 64
    # 7-40-40-3: its own width, biases as accumulators' start values, output layer N = 8
    assert macs(wk.WORKLOADS["c2"]) == 16 * 40 + 80 * 40 + 80 * 8
    # 4-16-16-3 and 8-16-16-16-3: output layer in fp32
    assert macs(wk.WORKLOADS["c1"]) == 16 * 16 + 32 * 16
    assert macs(_workload((8, 16, 16, 16, 3), 8, 1)) == 16 * 16 + 2 * 32 * 16


def test_alu_operations_with_the_kernels_gelu(bench):
    g = bench.GELU_OPS
    assert g == 8  # six Horner steps, the saturating subtraction, the last multiply-add
    ops = bench.alu_ops_per_px
    assert ops(wk.WORKLOADS["c4"], "fp16_tc", g) == 192 * 8 + 2 * 128 + 3 * 64
    assert ops(wk.WORKLOADS["c2"], "fp16_tc", g) == 80 * 8 + 2 * 80
    assert ops(wk.WORKLOADS["c5"], "fp16_tc", g) == 2 * 128
    assert ops(_workload((8, 16, 16, 16, 3), 8, 1), "fp16_tc", g) == 2 * 32 + 3 * 16
    assert ops(wk.WORKLOADS["c2"], "fp32", g) == 80 * 8 + 2000


def test_a_rows_counts_are_those_of_its_kernel(bench):
    wl = wk.WORKLOADS["c5"]
    px = 64 * wl.H * wl.W
    peaks = {"hbm_gbs": 6793.4, "bf16_tflops": 1956.0, "source": "measured"}
    for staging, macs in (("auto", bench.march_tensor_macs_per_px), ("tma", bench.executed_tensor_macs_per_px)):
        roof = bench.roofline_for(wl, "fp16_tc", 64, 1.0, peaks, 70.0, "measured", staging)
        assert roof["executed_tensor_flops_per_launch"] == 2.0 * macs(wl) * px
        assert roof["alu_bound"]["ops_per_px"] == 2 * 128
    assert bench.march_tensor_macs_per_px(wl) != bench.executed_tensor_macs_per_px(wl)


def test_sources_of_each_kernel(bench):
    assert "k_strip.cuh" in bench.kernel_sources("tc05_8x16x16x16x3_relu")
    assert "k_strip.cuh" in bench.kernel_sources("tc05_7x40x40x3_gelu_f32lat")
    assert "k_tcmarch.cuh" in bench.kernel_sources("tc05_7x64x64x3_relu")
    assert "k_tcmarch.cuh" in bench.kernel_sources("tc05_16x64x64x64x3_gelu_f32lat")
    for name in ("tc05_7x64x64x3_relu_tile", "tc05_4x16x16x3_relu_tma", "tc05_7x64x64x3_relu_lo8"):
        assert "k_tc.cuh" in bench.kernel_sources(name)
    assert bench.kernel_sources("fp32_generic") == bench.KERNEL_SOURCES["fp32"]
    assert bench.kernel_sources("idct_unpatchify_kernel") == ["k_idct.cu"]
    assert bench.kernel_source_hash("tc05_8x16x16x16x3_relu") != bench.kernel_source_hash("tc05_7x64x64x3_relu")

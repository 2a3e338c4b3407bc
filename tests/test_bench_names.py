"""The benchmark's lines name the kernel that ran and attach only traffic that was captured from it."""
import os

import bench
from paper_2107_06419_b200 import api

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_every_variant_has_a_kernel():
    for name in dir(api):
        if name.startswith("FLAT_VARIANT_") and name != "FLAT_VARIANT_AUTO":
            assert "kernel" in bench.kernel_name(getattr(api, name), 64), name
    assert bench.kernel_name(api.FLAT_VARIANT_TC2, 128) == "fused_d128_kernel"       # csrc/fused_tc2.cu hands it on
    assert bench.kernel_name(api.FLAT_VARIANT_TC2, 64) == "fused_tc2_kernel<2 tiles>"
    assert bench.kernel_name(api.FLAT_VARIANT_TC2_SPLIT8, 128).startswith("fused_tc2_kernel")


def test_traffic_has_its_capture():
    for (kernel, workload), (_, path) in bench.MEASURED_DRAM_TRAFFIC.items():
        text = open(os.path.join(ROOT, path)).read()
        assert kernel.split("<")[0] in text and workload in text, (kernel, workload)
    assert bench.traffic_fields("fused_d128_kernel", "a workload without a capture")["traffic"] is None

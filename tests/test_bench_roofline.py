"""The benchmark's rooflines: the interpreter's uses the capture of the kernel,
envs per warp and workload that ran, whatever the other options were; the
fused kernel's counts the bytes that the path cannot do without, not the band
snapshots that this way of painting reads."""
import pytest

import bench


@pytest.mark.parametrize("config", [2, 3])
def test_interpreter_roofline_finds_its_capture(config):
    prof = {"interpreter": (10.0, 5), "fused_raster_preprocess": (10.0, 5)}
    r = bench.interp_roofline(prof, 1e8, "k_interp_split", 32, config, 4096, 4)
    assert r["achieved"] > 0 and r["traffic"] > 0 and "this workload" in r["ratio_source"]
    assert bench.interp_roofline(prof, 1e8, "k_interp_batched", 32, config, 4096, 4)["achieved"] is None


def test_fused_roofline_counts_algorithmic_bytes():
    logged = 4096 * 1000.0
    r = bench.fused_roofline({"fused_raster_preprocess": (10.0, 5)}, logged, 2, 4096)
    assert r["algorithmic_bytes_per_env_step"] == 4 * 1000 + 16 + 8 * 84 * 84 + 1
    assert r["snapshot_bytes_per_env_step"] == 2 * 105 * 48

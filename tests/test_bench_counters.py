"""The DRAM traffic that the benchmark prints beside a kernel: counters of the kernel as it is, or none."""
import shutil

import pytest

import bench
import hts_workloads as wl


def test_counted_traffic_is_of_these_sources():
    cfg = wl.CONFIGS[bench.WORKLOAD]
    frames = cfg.N * cfg.C * cfg.H * cfg.W
    for kernel in bench.layer_macs(cfg):
        count = bench.dram_traffic(kernel)
        assert count is None or count == bench.DRAM_TRAFFIC[kernel][0]
    assert frames <= bench.DRAM_TRAFFIC["conv1"][0] <= 1.05 * frames


@pytest.mark.parametrize("change,kept", [("// a remark\n", True), ("static int changed;\n", False)])
def test_changed_source_has_no_counters(monkeypatch, tmp_path, change, kept):
    for _, source, _ in bench.DRAM_TRAFFIC.values():
        shutil.copy(f"{bench.CSRC}/{source}", tmp_path / source)
    recorded = {k: (v[0], v[1], bench.source_digest(tmp_path / v[1])) for k, v in bench.DRAM_TRAFFIC.items()}
    monkeypatch.setattr(bench, "CSRC", str(tmp_path))
    monkeypatch.setattr(bench, "DRAM_TRAFFIC", recorded)
    with open(tmp_path / "conv1_tc.cu", "a", encoding="utf-8") as f:
        f.write(change)
    assert (bench.dram_traffic("conv1") is not None) == kept and bench.dram_traffic("fc") is not None

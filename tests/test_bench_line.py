"""The benchmark's printed line on the CPU: short, whole in the fields that its
readers need, and with recorded DRAM traffic only where it was recorded for the
same sources and workload."""
import json

import bench


def full():
    cfg = {"workload": "w" * 200, "slots": 1 << 26, "load": 0.95, "n_insert": 63753421,
           "n_find": 1 << 26, "n_mixed": 1 << 24, "key_dist": "uniform u32 in [1, 2^32-3]",
           "seed": 2, "l2": "no flush: 512 MiB table and inputs exceed the 129 MB L2",
           "table": {"block_threads": 128, "bucket_slots": 16, "l2_persist": 0,
                     "max_evictions": 16, "placement": 0}}
    row = {"bound": "hbm", "achieved": 1558.4100000001, "peak": 6784.2, "unit": "GB/s",
           "frac": 0.22971234567, "traffic": 4627441920.0, "algorithmic_bytes": 4647169205,
           "avg_ms": 2.98198123456, "kernel": "k_insert_part+store<S=16>",
           "peak_source": "measured"}
    line = {"metric": bench.METRIC, "value": 25.913412345678, "unit": "Gops/s", "n_gpus": 1,
            "steps": 60, "warmup": 3, "ms_per_step": 5.697421234, "higher_is_better": True,
            "scaling": "weak", "vs_baseline": None, "dtype": "u32/u64", "data": "synthetic",
            "config": cfg,
            "phases": {**{f"{k}_{u}": 1.23456789012 for k in ("insert", "find", "mixed")
                          for u in ("gops", "ms")},
                       "kernel_ms_per_step": {k: 0.123456789 for k in
                                              ("find", "insert", "mixed", "evict", "maint", "claim")},
                       "paper_default_s32": {"x": 1.0}, "fused_mixed": {"rows": [1.0] * 500}},
            "roofline": {**row, "others": {k: row for k in ("find", "mixed", "claim")}},
            "cpu_baseline": {"value": 0.0045, "unit": "Gops/s", "cores": 1, "kind": "oracle",
                             "sample": "s" * 120, "host": {"cpus": 16, "model": "Neoverse-V2"}},
            "e2e": {"value": 19.9, "unit": "Gops/s", "h2d_bytes_per_step": 929457768,
                    "d2h_bytes_per_step": 483183821, "steps": 5, "api": "a" * 80,
                    "transfer": "t" * 90, "host_wall_gops": 19.9, "staged_gops": 17.9},
            "clocks": {"sm_mhz": 2070.0, "sm_max_mhz": 2070.0, "reasons": []},
            "gpu_launches": 480}
    extra = {"multi_table": {"batched_gops": 10.5, "plain_gops": 0.7, "note": "n" * 500},
             "serving": {"saturation": {"batched_gops": 9.1, "fifo_gops": 1.2},
                         "rates": [{"p50_ms": 0.17}] * 50},
             "insert_breakdown": {"rows": [0.1] * 2000}, "load_sweep": {"rows": [0.1] * 500},
             "hive32_key_only": {"insert_gops": 20.5, "find_gops": 55.1, "mixed_gops": 15.3}}
    return line, extra


def test_line_is_short_and_whole():
    line, extra = full()
    text = json.dumps(bench.result_line(line, extra))
    assert len(text) < 3000 and "\n" not in text
    d = json.loads(text)
    for k in ("metric", "unit", "n_gpus", "steps", "warmup", "higher_is_better", "scaling",
              "vs_baseline", "dtype", "data", "config", "clocks", "gpu_launches"):
        assert d[k] == line[k], k
    assert abs(d["value"] / line["value"] - 1) < 1e-5
    assert d["e2e"]["h2d_bytes_per_step"] == 929457768 and d["roofline"]["kernel"]
    assert d["legs"]["serving"] == {"batched_gops": 9.1, "fifo_gops": 1.2}
    assert bench.json.loads(json.dumps(bench.result_line(line, {})))["legs"] == {}


def test_recorded_traffic_needs_the_same_sources_and_workload(monkeypatch, tmp_path):
    f = tmp_path / "t.txt"
    f.write_text(f"# c\nkernel=k workload=w bytes_per_launch=5 source_sha={bench.source_sha()}\n"
                 "kernel=old workload=w bytes_per_launch=7 source_sha=0000\n")
    monkeypatch.setattr(bench, "TRAFFIC_FILE", str(f))
    assert bench.recorded_traffic("k", "w") == 5.0
    assert bench.recorded_traffic("k", "other") is None
    assert bench.recorded_traffic("old", "w") is None
    # a change in any of the sources ends it
    for name in bench.KERNEL_SRCS:
        monkeypatch.setattr(bench, "KERNEL_SRCS", [n for n in bench.KERNEL_SRCS if n != name])
        assert bench.recorded_traffic("k", "w") is None
        monkeypatch.undo()
        monkeypatch.setattr(bench, "TRAFFIC_FILE", str(f))


def test_insert_label_follows_the_path():
    assert bench.insert_kernel(1 << 26, 60_000_000, 16) == "k_insert_part+store<S=16>"
    assert bench.insert_kernel(1 << 25, 30_000_000, 16) == "k_ops<insert,S=16>"
    assert bench.insert_kernel(1 << 26, 1 << 20, 32) == "k_ops<insert,S=32>"

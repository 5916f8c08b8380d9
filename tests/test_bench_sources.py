"""The recorded ncu counters of each precision go stale with that precision's
kernel sources."""

import json

import bench


def test_counters_follow_their_own_sources(tmp_path, monkeypatch):
    mixed, fp64 = bench.kernel_hash(), bench.kernel_hash(sources=bench.FP64_SOURCES)
    assert mixed != fp64
    files = {f: f"int {f.split('.')[0]}();\n" for f in bench.FP64_SOURCES}
    base = bench.kernel_hash(files.__getitem__, bench.FP64_SOURCES)
    for f in files:
        assert bench.kernel_hash(dict(files, **{f: "int g();\n"}).__getitem__, bench.FP64_SOURCES) != base
    (tmp_path / "profiles").mkdir()
    monkeypatch.setattr(bench, "ROOT", str(tmp_path))
    monkeypatch.setattr(bench, "kernel_hash", lambda read=None, sources=bench.MIXED_SOURCES:
                        {bench.MIXED_SOURCES: mixed, bench.FP64_SOURCES: fp64}[sources])
    tab = {f"col_main|4096sq_{w}": {"kernel_hash": h, "dram_bytes_per_launch": 7}
           for w, h in (("mixed", mixed), ("fp64", fp64))}
    (tmp_path / "profiles" / "traffic.json").write_text(json.dumps(tab))
    assert [bench.load_traffic("col_main", "4096sq_" + w) for w in ("mixed", "fp64")] == [7, 7]
    tab["col_main|4096sq_fp64"]["kernel_hash"] = mixed
    (tmp_path / "profiles" / "traffic.json").write_text(json.dumps(tab))
    assert bench.load_traffic("col_main", "4096sq_fp64") is None

"""The benchmark's captured DRAM bytes: those of the shape when they were captured,
else the default shape's, named so, and neither when the kernel source differs."""
import hashlib
import json

import bench


def test_lookup(tmp_path, monkeypatch):
    (tmp_path / "k.cu").write_text("kernel")
    (tmp_path / "profiles").mkdir()
    digest = hashlib.sha256(b"kernel").hexdigest()[:16]
    entry = dict(source=["k.cu"], source_sha256_16=digest)
    (tmp_path / "profiles" / "traffic.json").write_text(json.dumps({
        "k_a_fp32_384": dict(entry, dram_bytes_per_launch=100),
        "k_a_fp32_384_p64": dict(entry, dram_bytes_per_launch=90),
        "k_b_fp32_384": dict(entry, dram_bytes_per_launch=80, source_sha256_16="0" * 16)}))
    monkeypatch.setattr(bench, "ROOT", str(tmp_path))
    assert bench.traffic_for("k_a_fp32_384", 0) == (100, "default")
    assert bench.traffic_for("k_a_fp32_384", 64) == (90, "param 64")
    assert bench.traffic_for("k_a_fp32_384", 67371200) == (100, "default")
    assert bench.traffic_for("k_b_fp32_384", 0) == (None, None)
    assert bench.traffic_for("k_c_fp32_384", 5) == (None, None)


def test_the_default_workloads_have_entries():
    with open(bench.os.path.join(bench.ROOT, "profiles", "traffic.json")) as fh:
        keys = json.load(fh)
    assert {"k_force3d+k_lb3d+k_phi3d_fp32_384", "k_force3d+k_lb3d+k_phi3d_iso_fp32_384", "k_march2d_x2_fp32_1024",
            "k_march2d_iso_x2_fp32_1024"} <= set(keys)

"""The Schwarz roofline of bench.py names the kernel that ran, and gives its DRAM
traffic only for the case it was captured for."""
import json
import os

import bench


def test_kernel_name_follows_block_and_storage():
    for prec in ("f32", "f16", "bf16", "f16n"):
        assert bench.sap_kernel((4, 4, 4, 4), prec) == bench.sap_kernel([8, 4, 4, 4], prec) == "k_sap_pair"
        assert bench.sap_kernel((4, 4, 4, 8), prec) == bench.sap_kernel((2, 2, 2, 2), prec) == "k_sap_phase"
    assert bench.sap_kernel((2, 2, 2, 2), "f64") == bench.sap_kernel((2, 4, 2, 2), "f64") == "k_sap_fine"
    assert bench.sap_kernel((4, 4, 4, 4), "f64") == "k_sap_phase"


def test_traffic_only_for_the_captured_case(tmp_path, monkeypatch):
    os.makedirs(tmp_path / "profiles")
    case = {"storage": "f32", "block": [4, 4, 4, 4], "sites": 1048576}
    (tmp_path / "src.cu").write_text("x")
    entry = {"bytes_per_launch": 5.0, "sources": ["src.cu"], "case": case,
             "source_sha256_16": "2d711642b726b044"}   # SHA-256 of "x"
    (tmp_path / "profiles" / "traffic.json").write_text(json.dumps({"k": entry}))
    monkeypatch.setattr(bench, "ROOT", str(tmp_path))
    assert bench.kernel_traffic("k", **case) == 5.0
    for other in ({"storage": "f16"}, {"block": [8, 4, 4, 4]}, {"sites": 131072}):
        assert bench.kernel_traffic("k", **{**case, **other}) is None
    for k, v in json.load(open(os.path.join(os.path.dirname(bench.__file__), "profiles", "traffic.json"))).items():
        assert {"block", "sites", "storage"} <= set(v["case"]) and v["case"]["sites"] == v["scaled_to_sites_per_launch"], k

"""bench.py takes counted figures of kernels (traffic, FP64-pipe operations) only for the sources they were counted on."""
import json

import bench


def _tables(tmp_path, monkeypatch, digest):
    (tmp_path / "profiles").mkdir()
    (tmp_path / "profiles" / "dram_traffic.json").write_text(json.dumps(
        {"source_sha256": digest, "kernels": {"update2d_fp64": {"bytes_per_cell": 7.0, "fp64_pipe_ops_per_cell": 5.0}}}))
    monkeypatch.setattr(bench, "source_hash", lambda sources=None: "now")
    monkeypatch.setattr(bench, "ROOT", str(tmp_path))


def test_figures_of_these_sources(tmp_path, monkeypatch):
    _tables(tmp_path, monkeypatch, "now")
    key = bench.FP64_KERNELS["update"][0]
    assert bench.traffic_per_cell(key) == 7.0
    assert bench.traffic_per_cell(key, figure="fp64_pipe_ops_per_cell") == 5.0
    assert bench.traffic_per_cell("rec2d_fp64", figure="fp64_pipe_ops_per_cell") is None


def test_figures_of_other_sources(tmp_path, monkeypatch):
    _tables(tmp_path, monkeypatch, "before")
    for key, _ in bench.FP64_KERNELS.values():
        assert bench.traffic_per_cell(key, figure="fp64_pipe_ops_per_cell") is None
        assert bench.traffic_per_cell(key) is None

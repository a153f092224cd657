"""The benchmark's figures from ncu records: a record counts only while every
source file its figures depend on is as it was captured.  Runs on a copy of the
records and sources."""
import hashlib
import json
import os
import shutil

import pytest

import bench

CSRC = os.path.join("paper_1307_2265_gb300", "csrc")
PROBE = {"dfma": {"ops_per_s": 5e11}}
FIGURES = {
    "fp64_alu.json": (lambda t: bench.fp64_alu_roofline(200.0, PROBE),
                      ["fp64_path.cu", "ppm_staged.cuh", "ppm_device.cuh", "exact64.cuh", "internal.cuh"]),
    "traffic.json": (lambda t: bench.measured_traffic(1e6, t["kernel"]),
                     ["fp32_path.cu", "ppm_device.cuh", "exact64.cuh", "internal.cuh", "mlp_layout.cuh", "tc05.cuh"]),
}


@pytest.mark.parametrize("name", sorted(FIGURES))
def test_a_changed_source_voids_the_record(name, tmp_path, monkeypatch):
    figure, sources = FIGURES[name]
    shutil.copytree(os.path.join(bench.ROOT, CSRC), tmp_path / CSRC)
    with open(os.path.join(bench.ROOT, "profiles", name)) as f:
        t = json.load(f)
    h = hashlib.sha256()
    for s in t["sources"]:
        h.update((tmp_path / s).read_bytes())
    t["sources_sha256_16"] = h.hexdigest()[:16]          # a record of the sources as they are
    (tmp_path / "profiles").mkdir()
    (tmp_path / "profiles" / name).write_text(json.dumps(t))
    monkeypatch.setattr(bench, "ROOT", str(tmp_path))
    assert figure(t) is not None
    for s in sources:
        p = tmp_path / CSRC / s
        was = p.read_bytes()
        p.write_bytes(was + b"\n")
        assert figure(t) is None, s
        p.write_bytes(was)
    assert figure(t) is not None

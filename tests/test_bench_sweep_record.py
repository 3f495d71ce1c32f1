"""What the benchmark's roofline record says about the sweep: the kernel by the
tile that ran, and a traffic figure only from a capture of the present sources and
of that tile."""
import json
import os
import re

import pytest

import bench

CSRC = os.path.join(bench.ROOT, "paper_2501_02245_gb300", "csrc")


@pytest.mark.parametrize("tuning,kernel", [
    ("1D line: window sweep", "k_sweep_line"), ("1D or empty: fixed shape", "k_sweep"),
    ("1D line: general sweep (tiles uneven over the SMs)", "k_sweep"),
    ("tile col_z2_g12_p16 (autotuned; tile timings (ms per pass pair): g16_v1_c1=7.5)", "k_sweep_col"),
    ("tile planes_wide (cached)", "k_sweep_planes"), ("tile p5_v2_c1 (autotuned; x)", "k_sweep2"),
    ("tile g4_v1_c1 (not tuned: no memory for a snapshot)", "k_sweep"), ("tile ring_w8_v32 (forced)", "k_sweep_ring")])
def test_the_kernel_is_named_by_the_tile(tuning, kernel):
    assert bench.sweep_kernel(tuning) == kernel


def test_the_source_list_holds_every_file_of_the_sweep():
    todo = [f for f in os.listdir(CSRC) if f.startswith("sweep") and f.endswith(".cu")]
    seen = set()
    while todo:
        f = todo.pop()
        if f in seen or not os.path.exists(os.path.join(CSRC, f)) or not f.endswith((".cu", ".cuh")):
            continue   # (the plain headers hold declarations)
        seen.add(f)
        todo += re.findall(r'#include "([^"]+)"', open(os.path.join(CSRC, f)).read())
    assert seen == set(bench.SWEEP_SOURCES)


def test_traffic_needs_the_present_sources_and_the_tile(tmp_path, monkeypatch):
    sha = bench.source_sha(["paper_2501_02245_gb300/csrc/" + f for f in bench.SWEEP_SOURCES])
    os.mkdir(tmp_path / "profiles")
    for f in bench.SWEEP_SOURCES:
        dst = tmp_path / "paper_2501_02245_gb300" / "csrc" / f
        dst.parent.mkdir(parents=True, exist_ok=True)
        dst.write_bytes(open(os.path.join(CSRC, f), "rb").read())
    monkeypatch.setattr(bench, "ROOT", str(tmp_path))
    rec = {"sweep_src_sha": sha, "tile": "planes", "dram_bytes_per_point": 9.0}

    def figure(**change):
        (tmp_path / "profiles" / "sweep_cylinder_f32.json").write_text(json.dumps(dict(rec, **change)))
        return bench.traffic_per_point("cylinder", "f32", "tile planes (cached)")

    assert figure() == 9.0
    assert figure(tile="p5_v2_c1") is None
    assert figure(sweep_src_sha="0") is None

"""What ties the recorded figures of bench.py to the code: the hash covers every
source that the stage kernels are built from, and both kernel forms are read."""
import os

import bench
from tests.test_lib_cpu import _ncu_csv


def test_hash_covers_what_the_stage_kernels_include(tmp_path, monkeypatch):
    files = {os.path.basename(f) for f in bench.stage_sources()}
    assert {"stage_f64.cu", "stage_f32.cu", "stage_f2x.cu", "stage_kernels.cuh", "stage_team.cuh", "stage_tuning.h",
            "f2x.cuh", "basis.h", "dependent_launch.cuh", "stage_launch.h", "hho_internal.h"} <= files
    before = bench.stage_source_sha()
    csrc = tmp_path / "paper_2505_15771_gb300" / "csrc"
    csrc.mkdir(parents=True)
    for f in bench.stage_sources():
        (csrc / os.path.basename(f)).write_bytes(open(f, "rb").read())
    monkeypatch.setattr(bench, "ROOT", str(tmp_path))
    assert bench.stage_source_sha() == before
    for name in ("stage_team.cuh", "basis.h", "hho_internal.h"):
        was = (csrc / name).read_bytes()
        (csrc / name).write_bytes(was + b"//\n")
        assert bench.stage_source_sha() != before
        (csrc / name).write_bytes(was)


def test_traffic_of_the_team_form_is_read(tmp_path):
    rows = [("void <unnamed>::team_kernel<f2x, 3, 1, 10>(StageArgsT<T1>)", 300.0, 180.0, 250.0),
            ("void <unnamed>::team_kernel<f2x, 3, 0, 10>(StageArgsT<T1>)", 999.0, 999.0, 90.0),
            ("void <unnamed>::team_kernel<double, (int)3, (int)1, (int)10>(StageArgsT<T1>)", 200.0, 100.0, 90.0)]
    _ncu_csv(tmp_path / "k3.csv", rows)
    rec = bench.write_traffic_record([(str(tmp_path / "k3.csv"), 40, 20, 3)], str(tmp_path / "out.json"))
    assert rec["f32x2_k3"]["dram_bytes_per_launch_mean"] == 480e6
    assert rec["k3"]["dram_bytes_per_launch_mean"] == 300e6

"""What bench.py takes from the committed counter summaries (host arithmetic, no GPU):
nothing once a source of the profiled kernel has changed, and no traffic at another size
than the captured one."""
import os
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
sys.path.insert(0, ROOT)

import bench  # noqa: E402


@pytest.mark.parametrize("path, needs", [
    (bench.PROFILE, ("kernels_fp32.cu", "sweep_pair.cuh", "sweep_mom.cuh", "wall_table.cuh", "biot_args.h", "biot_common.cuh")),
    (bench.PROFILE64, ("kernels_fp64.cu", "sweep_mom.cuh", "wall_table.cuh", "biot_args.h", "biot_common.cuh"))])
def test_hash_covers_every_source_of_the_launch(path, needs, monkeypatch, tmp_path):
    names = [os.path.basename(f) for f in bench.kernel_sources(path)]
    assert set(needs) | {"build.py"} <= set(names)
    before = bench.kernel_sha(path)
    for f in bench.kernel_sources(path):  # any one of them changes the hash
        changed = tmp_path / os.path.basename(f)
        changed.write_bytes(open(f, "rb").read() + b"\n")
        with monkeypatch.context() as m:
            m.setattr(bench, "kernel_sources", lambda p, f=f, c=str(changed), l=bench.kernel_sources(path): [c if x == f else x for x in l])
            assert bench.kernel_sha(path) != before, f


def test_counters_of_another_source_or_size_are_dropped(tmp_path, monkeypatch):
    profile = str(tmp_path / "p.md")
    monkeypatch.setitem(bench.KERNEL_UNIT, profile, "kernels_fp32.cu")
    sha = bench.kernel_sha(profile)

    def write(h):
        with open(profile, "w") as f:
            f.write(f"kernel_source_sha: {h}\ntraffic_bytes_per_cell: 64.5\ntraffic_cells: 16777216\n")
    write(sha)
    assert bench.profiled_traffic(4096 * 4096, profile) == pytest.approx(64.5 * 4096 * 4096)
    assert bench.profiled_traffic(2048 * 2048, profile) is None
    write("0" * 16)
    assert bench.profiled_traffic(4096 * 4096, profile) is None
    assert bench.profiled_traffic(4096 * 4096, str(tmp_path / "none.md")) is None


def test_coarse_sweeps_label_names_the_bound_of_the_precision():
    assert "64^2" in bench.coarse_sweeps_label(False, "fp32")
    assert "2048 cells" in bench.coarse_sweeps_label(False, "fp64")
    assert "16^2" in bench.coarse_sweeps_label(False, batched=True)
    assert "BIOT_OPT_SEGMENTS" in bench.coarse_sweeps_label(True, "fp64")

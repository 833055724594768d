"""The shared-memory tile of the watershed and the influence zones (csrc/iwpp_smemtile.cuh), compiled
for the host and run thread by thread (tests/host): no two unordered accesses to a pixel of the tile
but whole relaxed ones, each halo word has one writer, and the drain reaches the fixed point while
pixels beside a held tile change. Copies of the header with the fault put back are reported."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
HEADER = os.path.join(os.path.dirname(HERE), "paper_1605_00930_gb300", "csrc", "iwpp_smemtile.cuh")


def run_model(tmp_path, change=None):
    text = open(HEADER).read()
    if change:
        assert text.count(change[0]) == 1, "the line to change is not there once"
        text = text.replace(*change)
    (tmp_path / "iwpp_smemtile.cuh").write_text(text)
    for name, to in (("host_cta.h", "host_cta.h"), ("smem_engine.h", "iwpp_engine.cuh"), ("smem_tile.cpp", "smem_tile.cpp")):
        shutil.copy(os.path.join(HERE, "host", name), tmp_path / to)
    exe = tmp_path / "smem_tile"
    subprocess.check_call(["g++", "-std=c++17", "-O2", "-w", "-o", str(exe), str(tmp_path / "smem_tile.cpp")])
    return subprocess.run([str(exe)] + (["first"] if change else []), capture_output=True, text=True, timeout=300)


def test_no_races_and_the_fixed_point(tmp_path):
    r = run_model(tmp_path)
    assert r.returncode == 0, r.stdout + r.stderr


@pytest.mark.parametrize("change,bit", [
    (("p[i] = sm_ld_relaxed(prv + i);", "p[i] = prv[i];"), 2),     # another strip's row by plain loads
    (("sm_st_relaxed(row + 1, e);", "row[1] = e;"), 2),            # a plain store of a shared row
    (("const bool side = lane < 2 * kSmStrip;", "const bool side = true;"), 4),   # two lanes write a halo word
    (("__syncwarp();   // every lane has read the row", ""), 8),   # a vote alone before the row is written
])
def test_a_race_is_reported(tmp_path, change, bit):
    assert run_model(tmp_path, change).returncode & bit

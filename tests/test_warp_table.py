"""The table of csrc/warp_table.cuh keeps one record per key however the lanes
of a warp are scheduled between its barriers (run on the host, the lanes in
random order before every access)."""
import os
import subprocess

HERE = os.path.dirname(os.path.abspath(__file__))


def test_one_record_per_key_in_any_lane_order(tmp_path):
    exe = str(tmp_path / "warp_table")
    subprocess.run(["g++", "-O1", "-std=c++17", "-o", exe, os.path.join(HERE, "warp_table_host.cpp")], check=True)
    r = subprocess.run([exe, "2000"], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stdout + r.stderr

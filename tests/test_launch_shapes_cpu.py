"""Launch shapes (``csrc/launch_shapes.h``) on the host: the vocabulary projection's shared memory has room for the ring and for the
accumulator's rows at every row count and model width, and cross-attention takes its smaller blocks only where they are faster."""
import os
import subprocess

HERE = os.path.dirname(os.path.abspath(__file__))


def test_shapes_by_size(tmp_path):
    exe = tmp_path / "launch_shapes_check"
    subprocess.run(["g++", "-O1", "-std=c++17", os.path.join(HERE, "launch_shapes_check.cpp"), "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0 and r.stdout.strip() == "ok", r.stdout

"""Which steps are replayed as graphs (``csrc/step_graphs.h``), on the host: recorded once a size has come often enough to pay for it,
once per size, and launched kernel by kernel for good where a recording fails."""
import os
import subprocess

HERE = os.path.dirname(os.path.abspath(__file__))


def test_step_graphs(tmp_path):
    exe = tmp_path / "step_graphs_check"
    subprocess.run(["g++", "-O1", "-std=c++17", os.path.join(HERE, "step_graphs_check.cpp"), "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0 and r.stdout.strip() == "ok", r.stdout

"""The walking warps' bounded wait for a slot, compiled for the host from the
kernel's source (one OS thread per lane): a flag raised around the last look
never parts the warp, a slot written before is always taken, and one that is
never written is given up."""
import importlib.util
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))


def test_lanes_leave_together(tmp_path):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("g++ not available")
    spec = importlib.util.spec_from_file_location("emu_extract", os.path.join(HERE, "emu", "extract.py"))
    ex = importlib.util.module_from_spec(spec)
    spec.loader.exec_module(ex)
    src = open(os.path.join(ex.CSRC, "sweep.cu")).read()
    (tmp_path / "wait_device.h").write_text(ex._block(src, "__device__ __forceinline__ bool wait_slot("))
    exe = str(tmp_path / "run_wait")
    r = subprocess.run([gxx, "-std=c++17", "-O2", "-pthread", "-I", os.path.join(HERE, "emu"), "-I", str(tmp_path),
                        os.path.join(HERE, "emu", "run_wait.cpp"), "-o", exe], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-3000:]
    r = subprocess.run([exe, "2000"], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stdout + r.stderr[-2000:]

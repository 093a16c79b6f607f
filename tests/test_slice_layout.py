"""Row layout of the column slices on the host: tests/c_abi/slice_layout.cpp
linked to libtbcocg.so."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_offsets_do_not_depend_on_the_system_s_place(tmp_path):
    from paper_1002_1202_gb300 import _build_lib
    _build_lib.build()
    if shutil.which("g++") is None:
        pytest.skip("g++ not available")
    libdir = os.path.dirname(_build_lib.LIB)
    cuda = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(_build_lib._nvcc()))), "include")
    exe = str(tmp_path / "slice_layout")
    r = subprocess.run(["g++", "-std=c++17", "-O1", "-I", os.path.join(ROOT, "include"), "-I", cuda,
                        os.path.join(ROOT, "tests", "c_abi", "slice_layout.cpp"), "-o", exe, "-L", libdir, "-ltbcocg",
                        "-Wl,-rpath," + libdir], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    r = subprocess.run([exe], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0 and r.stdout.strip() == "ok", r.stdout + r.stderr

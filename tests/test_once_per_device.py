"""CPU check of csrc/once.h: a kernel's shared-memory limit is set once on each device, not once in
the process, and again where setting it failed."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2607_10983_gb300", "csrc")


def test_once_on_each_device(tmp_path):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no host C++ compiler")
    exe = str(tmp_path / "once_check")
    subprocess.run([cxx, "-std=c++17", "-O2", "-Wall", "-Werror", "-I", CSRC,
                    os.path.join(ROOT, "tests", "host", "once_check.cpp"), "-o", exe], check=True)
    # (device, what setting returns) -> (was it made, what comes back)
    script = [((0, 0), (1, 0)), ((0, 0), (0, 0)), ((1, 7), (1, 7)), ((1, 0), (1, 0)), ((1, 7), (0, 0)),
              ((63, 0), (1, 0)), ((63, 0), (0, 0)), ((64, 0), (1, 0)), ((64, 0), (1, 0)), ((0, 0), (0, 0))]
    out = subprocess.run([exe], input="\n".join(f"{d} {r}" for (d, r), _ in script), capture_output=True, text=True,
                         check=True).stdout
    assert [tuple(map(int, line.split())) for line in out.splitlines()] == [want for _, want in script]


def test_no_launcher_keeps_a_process_wide_flag():
    for name in os.listdir(CSRC):
        assert "static bool attr" not in open(os.path.join(CSRC, name)).read(), name

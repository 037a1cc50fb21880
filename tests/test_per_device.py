"""The per-device values behind launches that need a function attribute: each
device's are its own, made once, and a failure is not remembered (compiled for
the host and run here with device numbers; no GPU takes part)."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2405_01599_gb300", "csrc")

MAIN = r"""
#include "perdevice.cuh"
#include <cstdio>
int main() {
    xb::PerDevice<int> v;
    int out = -1, made = 0;
    auto make = [&](int device) { return [&made, device](int &t) { made++; t = 10 * device; return 0; }; };
    if (v.get(0, make(0), &out) != 0 || out != 0) return 1;
    if (v.get(1, make(1), &out) != 0 || out != 10) return 2;   // not the first device's
    if (v.get(0, make(7), &out) != 0 || out != 0 || made != 2) return 3;
    if (v.get(2, [](int &t) { t = 5; return -3; }, &out) != -3 || out != 0) return 4;
    if (v.get(2, make(2), &out) != 0 || out != 20) return 5;   // tried again
    return 0;
}
"""


def test_values_by_device(tmp_path):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no g++")
    src, exe = tmp_path / "main.cpp", tmp_path / "main"
    src.write_text(MAIN)
    subprocess.run([cxx, "-std=c++17", "-x", "c++", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    assert subprocess.run([str(exe)]).returncode == 0


def test_launch_limits_are_kept_by_device():
    """Every opt-in of the orthogonalisation's kernel is made for the device at hand."""
    src = open(os.path.join(CSRC, "ortho.cu")).read()
    body = src[src.index("int plan_launch("):src.index("int gs_run(")]
    assert "PerDevice<Limits>" in body and "cudaGetDevice" in body
    assert "static const" not in body

"""Kernels with more shared memory than a device allows by default, on a second
device of the same process and after a refused attempt (CPU: the launch functions
linked against a stand-in for the CUDA runtime, tests/device_limits_main.cpp)."""
import os
import subprocess

import pytest

import paper_2512_12094_gb300 as pp

HERE = os.path.dirname(os.path.abspath(__file__))
OBJECTS = ["pp_phase.cu.o", "pp_phase_rows.cu.o", "pp_merge.cu.o", "pp_kernels.cu.o"]


@pytest.fixture(scope="module")
def driver(tmp_path_factory):
    pp.build()
    built = [os.path.join(os.path.dirname(pp.__file__), "_build", o) for o in OBJECTS]
    if not all(os.path.exists(o) for o in built):
        pp.build(force=True)
    cuda = os.path.dirname(os.path.dirname(pp._nvcc())) or "/usr/local/cuda"
    exe = str(tmp_path_factory.mktemp("limits") / "limits")
    subprocess.run(["g++", "-O1", "-std=c++17", "-I", os.path.join(cuda, "include"),
                    os.path.join(HERE, "device_limits_main.cpp"), *built, "-o", exe], check=True)

    def run(*devices):
        out = subprocess.run([exe, *devices], capture_output=True, text=True, check=True, timeout=60).stdout
        return [(name, int(dev), int(status)) for name, dev, status in
                (line.split() for line in out.strip().split("\n"))]
    return run


def test_every_device_gets_its_limit(driver):
    rows = driver("0", "1", "0")
    assert {d for _, d, _ in rows} == {0, 1} and len(rows) == 3 * 37
    assert [r for r in rows if r[2] != 0] == []


def test_a_refused_attempt_is_not_remembered(driver):
    rows = driver("x0", "0", "1")
    assert len([r for r in rows if r[2] != 0]) == 1  # the first launch, once
    assert rows[0][2] != 0

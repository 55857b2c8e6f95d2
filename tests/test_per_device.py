"""Kernel attributes and occupancies belong to a device, not to the process
(csrc/per_device.h): a process with contexts on several devices sets a kernel's
shared-memory limit on each of them.  The header is built for the host with a
fake runtime of several devices; and every other file goes through it.
"""
import ctypes
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1303_4916_gb300", "csrc")


@pytest.fixture()
def lib(tmp_path):
    cxx, inc = shutil.which("g++"), "/usr/local/cuda/include"
    if not cxx or not os.path.isdir(inc):
        pytest.skip("no host C++ compiler or CUDA headers")
    out = str(tmp_path / "libpd.so")
    # -Bsymbolic: the fake runtime answers also where a real libcudart is in the process
    subprocess.run([cxx, "-O1", "-std=c++17", "-shared", "-fPIC", "-Wl,-Bsymbolic", "-I", CSRC, "-I", inc,
                    os.path.join(ROOT, "tests", "per_device_harness.cpp"), "-o", out], check=True)
    return ctypes.CDLL(out)


def test_each_device_is_asked_once(lib):
    for _ in range(3):
        for d in (0, 1, 2, 5, 63):
            lib.set_device(d)
            assert lib.ask_limit() == 0
            assert lib.ask_blocks() == d % 3
    for d in (0, 1, 2, 5, 63):
        assert lib.limit_calls(d) == 1 and lib.blocks_calls(d) == 1
    assert lib.limit_calls(3) == 0


def test_a_failure_is_not_kept_and_devices_beyond_the_table_are_asked_each_time(lib):
    lib.set_device(4)
    lib.set_fail(1)
    assert lib.ask_limit() == -1 and lib.ask_blocks() == -1
    lib.set_fail(0)
    assert lib.ask_limit() == 0 and lib.ask_blocks() == 1
    assert lib.limit_calls(4) == 2
    lib.set_device(100)
    assert [lib.ask_blocks() for _ in range(3)] == [1, 1, 1] and lib.blocks_calls(100) == 3


def test_no_other_file_asks_the_runtime_itself():
    for f in sorted(os.listdir(CSRC)):
        if f.endswith((".cu", ".cuh", ".h")) and f != "per_device.h":
            with open(os.path.join(CSRC, f)) as fh:
                text = fh.read()
            for call in ("cudaFuncSetAttribute", "cudaOccupancyMaxActiveBlocks"):
                assert call not in text, (f, call)

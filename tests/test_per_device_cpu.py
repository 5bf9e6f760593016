"""Kernel attributes and cluster counts belong to one device: what the launch
code keeps of them is kept per device (csrc/per_device.h), never for the
process.  Checked with a host build of the table and made-up devices."""

import ctypes
import glob
import os
import re
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2310_00226_gb300", "csrc")

SOURCE = """
#include "per_device.h"
static sem3d::PerDevice table;
static int calls;
extern "C" int n_calls() { return calls; }
extern "C" int get(int device, int value, int status) {  // -> the number, or -status
  int out = 0;
  const int st = table.get(device, out, [&](int& o) { ++calls; o = value; return status; });
  return st ? -st : out;
}
"""


@pytest.fixture
def table(tmp_path):
    (tmp_path / "t.cpp").write_text(SOURCE)
    subprocess.run(["g++", "-std=c++17", "-shared", "-fPIC", "-I", CSRC, str(tmp_path / "t.cpp"), "-o",
                    str(tmp_path / "t.so")], check=True)
    return ctypes.CDLL(str(tmp_path / "t.so"))


def test_each_device_is_asked_once(table):
    assert [table.get(d, 10 + d, 0) for d in (0, 1, 63)] == [10, 11, 73]
    assert table.n_calls() == 3
    assert [table.get(d, 99, 0) for d in (63, 0, 1)] == [73, 10, 11]  # kept
    assert table.n_calls() == 3


def test_failures_and_ordinals_beyond_the_table_are_not_kept(table):
    assert table.get(5, 1, 7) == -7
    assert table.get(5, 8, 0) == 8
    assert [table.get(64, v, 0) for v in (3, 4)] == [3, 4]
    assert table.get(-1, 6, 0) == 6
    assert table.n_calls() == 5


def test_launch_code_keeps_no_attribute_state_for_the_process():
    # next to every cudaFuncSetAttribute there is a PerDevice, and no static
    # flag or counter besides it
    for path in glob.glob(os.path.join(CSRC, "*.cu")):
        text = open(path).read()
        for m in re.finditer("cudaFuncSetAttribute", text):
            assert "on_device(" in text[max(0, m.start() - 300):m.start()], path
        assert not re.search(r"^\s+static std::atomic", text, re.M), path

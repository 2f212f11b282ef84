"""Host-side units of the library's launch code, compiled with nvcc and run without a GPU."""
import os
import subprocess

import pytest

from paper_2211_13028_gb300 import build as B

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def units(tmp_path_factory):
    exe = str(tmp_path_factory.mktemp("units") / "host_units")
    cmd = [B._nvcc(), *B.ARCH, "-std=c++17", "-cudart", "shared", "-I", B.INCLUDE, "-I", B.CSRC,
           os.path.join(HERE, "host_units.cu"), os.path.join(HERE, "host_units_runtime.c"), "-o", exe]
    r = subprocess.run(cmd, capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    return exe


def _run(units, check):
    r = subprocess.run([units, check], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0, r.stdout + r.stderr


def test_splits_of_one_branch_are_not_seen_by_another(units):
    # a branch's stream is ordered after the call's stream, not after the other branches', so a split that
    # another branch's kernel writes may not have been written when this one's reads it
    _run(units, "split_visibility")


def test_kernel_limits_and_sm_counts_are_each_devices_own(units):
    # handles on several devices of a process launch the same kernels
    _run(units, "per_device")


def test_expansions_are_split_into_the_parts_that_end_first(units):
    # as many items as 8 an SM: 1600 x 4992 out of 39 was 1092 items that converted 7 tiles 156 times each
    _run(units, "expand_parts")

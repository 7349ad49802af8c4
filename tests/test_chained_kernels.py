"""Kernels that may start while the kernel before them still runs (programmatic
dependent launch) read only the loaded layout as read-only data: the wait orders
ordinary accesses, and .nc loads need memory that nothing writes while the
reading kernel is resident."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1410_8043_gb300", "csrc")
# arrays that esspt_mf_load writes, and no kernel of a clock
LAYOUT = {"part", "items", "uoff", "item_rep", "hot_item", "item_cnt", "popular", "heavy"}


def _code(name):
    text = open(os.path.join(CSRC, name)).read()
    return re.sub(r"//[^\n]*", "", re.sub(r"/\*.*?\*/", "", text, flags=re.S))


def _chained():
    """{kernel: (parameters, body)} of the kernels that wait for the one before."""
    out = {}
    for name in sorted(os.listdir(CSRC)):
        if not name.endswith((".cu", ".cuh")):
            continue
        for f in re.finditer(r"__global__\s+void\s+(?:__launch_bounds__\([^)]*\)\s*)?(\w+)\(([^)]*)\)\s*\{(.*?)\n\}\n",
                             _code(name), flags=re.S):
            if "await_previous_kernel" in f[3]:
                out[f[1]] = f[2], f[3]
    return out


def _check_body(body):
    assert "ldg_f2x2_if" not in body and ".nc" not in body
    for arg in re.findall(r"__ldg\(([^;]*)", body):
        arrays = re.findall(r"\b[ac]\.(?!n_)(\w+)", arg.split(")")[0])
        assert arrays and set(arrays) <= LAYOUT, arg[:60]


def test_every_chained_launch_waits():
    launched = set()
    for name in os.listdir(CSRC):
        if name.endswith(".cu"):
            launched |= set(re.findall(r"launch_chained\((\w+)", _code(name))) - {"kernel"}
    assert launched | {"sgd_stream_kernel"} == set(_chained())


@pytest.mark.parametrize("kernel", ["sgd_stream_kernel", "clock_merge_kernel", "schedule_kernel", "copy_rows_kernel",
                                    "get_rows_kernel", "inc_rows_kernel"])
def test_reads_of_chained_kernels(kernel):
    params, body = _chained()[kernel]
    assert "__restrict__" not in params
    assert body.count("await_previous_kernel") == 1
    _check_body(body)


@pytest.mark.parametrize("header", ["copy_idle.cuh", "schedule.cuh"])
def test_reads_of_their_helpers(header):
    _check_body(_code(header))

"""Kernels launched as programmatic dependents live while the kernel before them
on the stream still writes: each waits for it before it touches memory, and none
reads through the read-only path or promises (by __restrict__ on a parameter)
that nothing else writes what it reads."""
import glob
import os
import re

import pytest

from paper_2607_14431_gb300 import build

WAITS = ("after_previous()", "split_begin(", "merge_partials<")


def _code():
    text = "\n".join(open(f).read() for f in sorted(glob.glob(os.path.join(build.CSRC, "*.cu*"))))
    return re.sub(r"//[^\n]*", "", text)


def _kernels(code):
    """(name, parameters, body) of every __global__ function."""
    for m in re.finditer(r"__global__\s+void\s+(?:__launch_bounds__\([^)]*\)\s*)?(\w+)\s*\(", code):
        end = code.index(") {", m.end())
        depth, i = 1, end + 3
        while depth:
            depth += {"{": 1, "}": -1}.get(code[i], 0)
            i += 1
        yield m.group(1), code[m.end():end], code[end:i]


def test_every_kernel_is_seen():
    code = _code()
    assert len(list(_kernels(code))) == code.count("__global__") >= 20


@pytest.mark.parametrize("name,params,body", list(_kernels(_code())), ids=[k[0] for k in _kernels(_code())])
def test_kernel_waits_and_reads_coherently(name, params, body):
    assert "__restrict__" not in params
    plain = re.search(name + r"\s*(<[^<>]*>)?\s*<<<", _code())
    assert plain or any(w in body for w in WAITS), "launched as a dependent without a wait"


def test_no_load_takes_the_read_only_path():
    code = _code()
    assert "__ldg(" not in code and "ld.global.nc" not in code

"""The kernels launched to overlap the one before (mtpt.cu `launch`), by their
source: each waits for that kernel before it reads what a kernel may have
written."""
import os
import re

import pytest

from paper_2204_03756_gb300 import build


def _source(name):
    with open(os.path.join(build.SRC_DIR, name)) as f:
        return re.sub(r"//[^\n]*", "", f.read())


def _kernel(src, name):
    """(parameter list, body) of the kernel's definition."""
    m = re.search(r"\b%s\s*\(" % name, src)
    end = m.end()
    depth = 1
    while depth:
        depth += {"(": 1, ")": -1}.get(src[end], 0)
        end += 1
    body = src.index("{", end)
    stop, depth = body + 1, 1
    while depth:
        depth += {"{": 1, "}": -1}.get(src[stop], 0)
        stop += 1
    return src[m.end():end - 1], src[body:stop]


KERNELS = sorted(set(re.findall(r"\blaunch\((k_\w+)", _source("mtpt.cu"))))


def test_the_step_kernels_are_found():
    assert {"k_scan", "k_gather", "k_rowsum_f32", "k_exchange_f64", "k_adj_exchange"} <= set(KERNELS)


@pytest.mark.parametrize("name", KERNELS)
def test_indexes_pass_through_the_wait(name):
    """A load whose address does not come out of the wait may be moved ahead of
    it: a kernel that reads through pointers to const takes its index from
    ordered_index()."""
    params, body = _kernel(_source("kernels.cuh"), name)
    if "ordered_index()" not in body:
        assert "after_previous()" in body
        assert not re.search(r"\bconst\b[^,]*\*", params)


CONSTANTS = {"corners", "exp_table"}     # written before the first kernel of a run starts


@pytest.mark.parametrize("name", KERNELS)
def test_read_only_pointers_are_constants(name):
    """The read-only path wants memory that nothing writes while the kernel
    lives, and an overlapping kernel is alive while the one before it writes."""
    params, _ = _kernel(_source("kernels.cuh"), name)
    assert set(re.findall(r"\bconst\b[^,]*\*\s*__restrict__\s+(\w+)", params)) <= CONSTANTS


def test_read_only_loads_are_of_constants():
    src = _source("kernels.cuh")
    assert set(re.findall(r"__ldg\((\w+)", src)) <= CONSTANTS
    assert not re.search(r"\bld\.[\w.]*\.nc\b", src)
    # nor in the device functions that the kernels share
    for params in re.findall(r"__device__[^;{]*?\(([^;{]*)\)\s*\{", src):
        names = set(re.findall(r"\bconst\b[^,]*\*\s*__restrict__\s+(\w+)", params))
        assert names <= CONSTANTS | {"table"}, names      # (table: in shared memory)


def test_no_kernel_lets_the_next_one_start_early():
    """Blocks that wait on the SMs while a kernel of a few blocks an SM still starts
    spread unevenly: the next kernel may start when this one's blocks have ended."""
    assert "launch_dependents" not in _source("kernels.cuh")

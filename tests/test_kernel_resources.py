"""Registers and spills of kernels whose speed hangs on them, as the compiler reports them (no GPU):
64 registers let four blocks of 256 threads share an SM, 80 three; a spilled register costs a trip
through local memory in the inner loop."""
import concurrent.futures
import os
import re
import subprocess

import pytest

from paper_1812_02091_gb300 import _build

SOURCES = ("k_phase1.cu", "k_sparse.cu", "k_sparse_b.cu", "k_within_b.cu")


def _compile(source):
    """{mangled kernel name: (registers, bytes of spill stores and loads)} of one translation unit."""
    cmd = [_build.nvcc()] + _build.ARCH + [f for f in _build.NVCC_FLAGS if f != "-lineinfo"] + [
        "-Xptxas", "-v", "-c", os.path.join(_build.CSRC, source), "-o", os.devnull]
    text = subprocess.run(cmd, capture_output=True, text=True, check=True).stderr
    return {m[1]: (int(m[4]), int(m[2]) + int(m[3])) for m in re.finditer(
        r"entry function '(\S+)'.*?(\d+) bytes spill stores, (\d+) bytes spill loads.*?Used (\d+) registers", text, re.S)}


@pytest.fixture(scope="module")
def kernels():
    with concurrent.futures.ThreadPoolExecutor() as pool:
        return dict(zip(SOURCES, pool.map(_compile, SOURCES)))


@pytest.mark.parametrize("source,kernel,registers", [
    ("k_sparse.cu", r"k_revILi\dELi[12]ELi4E", 64), ("k_sparse_b.cu", r"k_rev_bILi\dELi[12]ELi4E", 64),
    ("k_within_b.cu", r"k_rev_within_bILi\dELi[12]ELi4E", 64)])
def test_blocks_per_sm(kernels, source, kernel, registers):
    found = {n: r for n, (r, _) in kernels[source].items() if re.search(kernel, n)}
    assert found and max(found.values()) <= registers, found


@pytest.mark.parametrize("kernel", [r"k_dist_fp32E", r"k_dist_fp32_bE"])
def test_no_spills(kernels, kernel):
    found = {n: b for n, (_, b) in kernels["k_phase1.cu"].items() if re.search(kernel, n)}
    assert len(found) == 1 and not any(found.values()), found

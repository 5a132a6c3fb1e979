"""The benchmark's kernel version (the key under which measured DRAM traffic is kept) changes with every
source of the dslash kernels that the solves launch, and with no other."""
import os
import shutil
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1611_00298_gb300", "csrc")
sys.path.insert(0, ROOT)

import bench  # noqa: E402


@pytest.mark.parametrize("name,changes", [
    ("dslash_pair.cuh", True), ("dslash_impl.cuh", True), ("dslash_bulk.cuh", True), ("dslash_pipe.cuh", True),
    ("field.cuh", True), ("pair_op.h", True), ("dslash_pair_p32.cu", True), ("heatbath.cu", False), ("md.cu", False)])
def test_version_follows_the_kernel_sources(tmp_path, name, changes):
    copy = tmp_path / "csrc"
    shutil.copytree(CSRC, copy)
    assert bench.kernel_version(str(copy)) == bench.kernel_version()
    with open(copy / name, "a") as f:
        f.write("// edited\n")
    assert (bench.kernel_version(str(copy)) != bench.kernel_version()) == changes

"""A handle's dressing workspace is as large as the GPU has room for: the packed operands of the FP64 products
(750 MiB at 82 orbitals) are left out rather than the handle refused.  CPU check of that choice against a
fake allocator, and that the handle makes it after its other allocations."""
import os
import re
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))


def test_largest_size_that_fits(tmp_path):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no host C++ compiler")
    exe = str(tmp_path / "alloc_largest_check")
    subprocess.run([cxx, "-std=c++17", "-O1", os.path.join(HERE, "native", "alloc_largest_check.cpp"), "-o", exe],
                   check=True)
    res = subprocess.run([exe], capture_output=True, text=True)
    assert res.returncode == 0, res.stderr
    assert res.stdout.strip() == "ok"


def test_workspace_is_the_last_allocation_of_a_handle():
    src = open(os.path.join(os.path.dirname(HERE), "paper_2606_04186_gb300", "csrc", "host.cu")).read()
    init = src[src.index("int qflow_init("):]
    init = init[:init.index("\n}\n")]
    at = init.index("alloc_largest(")
    assert not re.search(r"cudaMalloc\(&c->(?!dwork)|dalloc\(&c->", init[at:])

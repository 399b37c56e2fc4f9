"""The sources that decide whether a stored traffic figure still belongs to a
kernel class: every file the compiler reads for the class's translation units."""
import os
import shutil
import subprocess

import pytest

import bench
from paper_2601_15401_gb300 import build as B


@pytest.mark.parametrize("group,units", [("ntt", sorted(f for f in os.listdir(B.CSRC) if f.startswith("ntt") and f.endswith(".cu"))),
                                         ("rns", ["rns.cu", "tensor_fixed.cu"])])
def test_every_file_of_a_class_counts(group, units):
    listed = bench.kernel_sources(group)
    assert set(units) <= set(listed) and set(units) <= set(B.SOURCES)
    nvcc = B.nvcc()
    if not shutil.which(nvcc):
        pytest.skip("no nvcc")
    read = set()
    for u in units:
        out = subprocess.run([nvcc, *B.ARCH, "-std=c++17", "-M", os.path.join(B.CSRC, u)], capture_output=True,
                             text=True, check=True).stdout
        paths = [os.path.realpath(x) for x in out.replace("\\\n", " ").split()[2:]]
        read |= {os.path.basename(x) for x in paths if os.path.dirname(x) == os.path.realpath(B.CSRC)}
    assert read | set(units) == set(listed)

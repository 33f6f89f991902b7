"""Index arithmetic and launch rules of the CUDA library (csrc/rules.cuh), compiled
for the host: the same functions as the kernels' and the library's host code."""
import ctypes
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2401_03180_gb300", "csrc")


@pytest.fixture(scope="module")
def rules(tmp_path_factory):
    """compile(body): a shared library of the C functions in body, over rules.cuh."""
    def compile_(body):
        d = tmp_path_factory.mktemp("rules")
        src, lib = d / "r.cpp", d / "r.so"
        src.write_text('#include "rules.cuh"\nusing namespace mdg;\nextern "C" {\n' + body + "\n}\n")
        subprocess.check_call(["g++", "-std=c++17", "-shared", "-fPIC", "-Wall", "-Werror", f"-I{CSRC}", "-o", str(lib), str(src)])
        return ctypes.CDLL(str(lib))
    return compile_


@pytest.mark.parametrize("d,k", [(0, 0), (7, 7), (8, None), (65_535, None), (65_536, None), (65_543, None), (1 << 20, None)])
def test_self_cluster_compares_the_whole_difference(rules, d, k):
    """A j-cluster of the own cell is the diagonal only as one of the super-cluster's
    up to eight i-clusters, however many clusters the cell holds."""
    lib = rules("unsigned f(int own, unsigned jc, unsigned fc) { return self_cluster(own != 0, jc, fc); }\n"
                "unsigned none() { return kNoSelf; }")
    for fc in (0, 3, 1 << 24):
        assert lib.f(1, fc + d, fc) == (lib.none() if k is None else k)
        assert lib.f(0, fc + d, fc) == lib.none()
    assert lib.none() >= 8

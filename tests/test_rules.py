"""Index arithmetic and launch rules of the CUDA library (csrc/rules.cuh), compiled
for the host: the same functions as the kernels' and the library's host code."""
import ctypes
import os
import subprocess

import numpy as np
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


@pytest.mark.parametrize("slot", [0, 8, 1 << 20, 1 << 24, (1 << 24) + 4096, 1 << 25, (1 << 30) - 8])
def test_padding_is_out_of_reach_of_padding(rules, slot):
    """Pads of a cluster, as the mixed force kernel stages them on the i side, against
    the same cluster's and other cells' pads on the j side, in 32 bits: never within
    the largest cutoff (1,000 nm), though the j side's coincide from slot 2^24 on."""
    lib = rules("float x(int s) { return (float)pad_x(s); }\n"
                "float staged(float x, float q) { return staged_x(x, q); }\n"
                "float charge() { return kPadCharge; }\nfloat far_() { return (float)kPadFar; }")
    for f in (lib.x, lib.staged, lib.charge, lib.far_):
        f.restype = ctypes.c_float
    lib.staged.argtypes = [ctypes.c_float, ctypes.c_float]
    pads = np.array([lib.x(slot + k) for k in range(8)], np.float32)
    assert (len(np.unique(pads)) < 8) == (slot >= 1 << 24)
    i = np.array([lib.staged(v, lib.charge()) for v in pads], np.float32)
    y = np.float32(lib.far_())
    for shift in (0.0, 1.2, -8192.0, 1.0e6):
        dx = i[:, None] - (pads + np.float32(shift))[None]
        dy = y - (y + np.float32(shift))
        r2 = dx * dx + np.float32(2) * dy * dy
        assert np.isfinite(r2).all() and r2.min() > 1.0e6 ** 2
    assert lib.staged(ctypes.c_float(3.5), ctypes.c_float(0.0)) == 3.5          # a neutral atom stays where it is
    assert lib.staged(ctypes.c_float(3.5), ctypes.c_float(2.0)) == 3.5


# (FP64, hybrid, warps, type states, blocks): the shapes that the interface has always accepted
PINS = [(0, 0, 4, 2, 6), (0, 0, 8, 2, 3), (0, 0, 12, 2, 2), (0, 0, 4, 46, 4), (0, 0, 8, 46, 2), (0, 0, 12, 46, 1),
        (0, 0, 8, 128, 1), (0, 1, 4, 28, 4), (0, 1, 12, 10, 1),
        (1, 0, 4, 28, 3), (1, 0, 4, 30, 3), (1, 0, 4, 31, 2), (1, 0, 4, 57, 2), (1, 0, 4, 58, 1), (1, 0, 4, 94, 1),
        (1, 0, 8, 2, 1), (1, 1, 4, 14, 3), (1, 1, 4, 15, 2), (1, 1, 4, 51, 2), (1, 1, 4, 52, 1), (1, 1, 8, 2, 1)]


@pytest.mark.parametrize("fp64,hyb,warps,n_ts,blocks", PINS)
def test_pinned_blocks_per_sm_stay_accepted(rules, fp64, hyb, warps, n_ts, blocks):
    lib = rules("int f(int d, int h, int w, int n) { return pair_pin_limit(d != 0, h != 0, w, n); }")
    assert lib.f(fp64, hyb, warps, n_ts) == blocks


@pytest.mark.parametrize("fused,sc_cap,per_sm,blocks", [(1, 32_768, 1, 152), (1, 32_768, 8, 1216), (1, 32_768, 16, 2432), (1, 300, 2, 300),
                                                        (1, 1, 16, 1), (0, 40_000, 1, 152), (0, 40_000, 16, 2432), (0, 40_000, 64, 5000)])
def test_list_blocks_per_sm_set_the_grid_of_either_build(rules, fused, sc_cap, per_sm, blocks):
    lib = rules("int f(int fused, int sc, int per, int sm) { return list_grid(fused != 0, sc, per, sm); }")
    assert lib.f(fused, sc_cap, per_sm, 152) == blocks


# (filled cells, atoms, capacity in super-clusters, one kernel)
@pytest.mark.parametrize("cells,atoms,sc_cap,one", [
    (125, 30_000, 3_860, True), (729, 199_773, 25_611, True), (1331, 240_000, 31_166, True),      # liquids
    (3_375, 3_375, 3_376, True), (4_913, 4_913, 4_914, False), (27_000, 27_000, 27_001, False),   # an atom a cell
    (1_728, 13_824, 3_241, True), (15_625, 125_000, 29_298, False),                               # eight a cell
    (3_375, 91_125, 14_344, True), (6_859, 185_193, 29_151, False),                               # 27 a cell
    (400, 4_000, 22_901, True),                                                                   # a batch of molecules
    (2_000, 300_000, 39_013, False), (600, 3_000, 33_976, False)])                                # beyond the capacity
def test_lists_of_few_super_clusters_are_built_by_one_kernel(rules, cells, atoms, sc_cap, one):
    lib = rules("int f(int cells, int atoms, int cap) { return list_in_one_kernel(cells, atoms, cap); }")
    assert bool(lib.f(cells, atoms, sc_cap)) == one


# (atoms, replicas, type states, a table of the rates) at 152 multiprocessors
@pytest.mark.parametrize("atoms,replicas,n_ts,table", [
    (1_999_998, 1, 43, True), (199_773, 1, 43, True), (1_400_000, 256, 43, True), (77_793, 1, 43, True),   # large samples
    (77_792, 1, 43, False), (30_000, 1, 43, False),                                                         # few blocks per SM
    (80_000, 8_000, 43, False), (688_000, 8_000, 43, True), (687_999, 8_000, 43, False),                    # small replicas
    (1 << 30, 1 << 29, 128, False)])
def test_rates_come_from_a_table_no_larger_than_the_sample(rules, atoms, replicas, n_ts, table):
    lib = rules("int f(long long n, long long r, int ts, int sm) { return rates_by_table(n, r, ts, sm); }")
    lib.f.argtypes = [ctypes.c_longlong, ctypes.c_longlong, ctypes.c_int, ctypes.c_int]
    assert bool(lib.f(atoms, replicas, n_ts, 152)) == table

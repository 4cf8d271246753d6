"""The node lists of a tournament hold every node of every level
(csrc/tree_nodes.h), and trees whose levels round up often still give the
oracle's factors."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

import workloads as wl

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2010_05975_gb300", "csrc")


@pytest.fixture(scope="module")
def capacity(tmp_path_factory):
    d = tmp_path_factory.mktemp("tree")
    (d / "t.cpp").write_text('#include "tree_nodes.h"\n'
                             'extern "C" long long capacity(int m, int h) { return (long long)lu::tree_capacity(m, h); }\n')
    subprocess.run(["g++", "-std=c++17", "-fPIC", "-shared", f"-I{CSRC}", str(d / "t.cpp"), "-o", str(d / "t.so")], check=True)
    f = ctypes.CDLL(str(d / "t.so")).capacity
    f.restype = ctypes.c_longlong
    return f


@pytest.mark.parametrize("h", [1, 3, 128, 512])
def test_lists_hold_all_levels_of_every_tree(capacity, h):
    """Every factorization step's tree, whose first level has at most
    ceil((m - k) / h) nodes: all levels one after another, and two levels in
    two halves."""
    for first in list(range(1, 3000)) + [4097, 8193, 65537, 100001]:
        m = (first - 1) * h + 1
        cap = capacity(m, h)
        total, n = 0, first
        while True:
            total += n
            if n == 1:
                break
            n = (n + 1) // 2
        assert cap >= total and cap // 2 >= first, (first, cap, total)


@pytest.mark.gpu
@pytest.mark.parametrize("dtype", ["f64", "f32"])
@pytest.mark.parametrize("m,n,b,h", [(2049, 40, 32, 128), (2100, 33, 32, 128), (4200, 48, 16, 128), (20000, 64, 32, 128),
                                     (1090, 70, 8, 32)])
def test_trees_with_rounded_up_levels(oracle_mod, dtype, m, n, b, h):
    """17, 33 and 157 first-level nodes (their trees have more than 2 (N + 1)
    nodes), steps that go through them, and what follows."""
    from tests.gpu_util import cuda_or_fail, lib
    torch = cuda_or_fail()
    g = lib()
    A = wl.matrix_uniform(m, n, seed=m)
    if dtype == "f32":
        A = A.astype(np.float32)
    LUo, po, io = (oracle_mod.lu_factor if dtype == "f64" else oracle_mod.lu_factor_f32)(A, b=b, h=h)
    d = torch.from_numpy(A.copy()).cuda()
    for _ in range(2):
        d.copy_(torch.from_numpy(A))
        piv, info = g.lu_factor_ex(d, b=b, h=h) if dtype == "f64" else g.lu_factor_f32(d, b=b, h=h)
        np.testing.assert_array_equal(piv.cpu().numpy(), po)
        assert int(info.cpu()[0]) == io
        np.testing.assert_array_equal(d.cpu().numpy(), LUo)

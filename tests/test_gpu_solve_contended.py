"""Substitutions beside other work that holds the SMs: the chain of the
binary32 substitution then takes over tasks that no other CTA has started
(csrc/getrs.cu), in the same order of operations."""
import numpy as np
import pytest

import workloads as wl
from tests.gpu_util import cuda_or_fail, lib

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,nrhs", [(1100, 8), (3001, 16), (5000, 32), (9700, 5)])
@pytest.mark.parametrize("chol", [False, True])
def test_same_bits_beside_other_work(n, nrhs, chol):
    torch = cuda_or_fail()
    lib()
    from paper_2010_05975_gb300 import api
    L = torch.from_numpy(wl.matrix_uniform(n, n, seed=n).astype(np.float32)).cuda() / n
    L.diagonal().add_(1.0)
    B = torch.from_numpy(wl.matrix_normal(n, nrhs, seed=n + 1).astype(np.float32)).cuda()
    piv = torch.arange(n, dtype=torch.int32, device="cuda")

    def solve():
        X = B.clone()
        api.chol_solve(L, X) if chol else api.lu_solve_f32(L, piv, X)
        return X

    want = solve()
    side = torch.cuda.Stream()
    M = torch.ones(8192, 8192, dtype=torch.bfloat16, device="cuda")
    O = torch.empty_like(M)
    torch.cuda.synchronize()
    for _ in range(3):
        with torch.cuda.stream(side):
            for _ in range(10):
                torch.matmul(M, M, out=O)
        assert torch.equal(solve(), want)
    torch.cuda.synchronize()

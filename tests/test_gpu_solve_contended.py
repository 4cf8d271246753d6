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


@pytest.mark.parametrize("n,nrhs", [(900, 3), (3000, 16), (10000, 40)])
def test_chain_wait_runs_out_then_recovers(n, nrhs):
    """A wait that nothing ends: the kernel drains within the deadline and the
    cluster's remaining steps, the call says so, and the next one is right."""
    import time
    torch = cuda_or_fail()
    g = lib()
    from paper_2010_05975_gb300 import api
    L = torch.from_numpy(wl.matrix_uniform(n, n, seed=n).astype(np.float32)).cuda() / n
    L.diagonal().add_(1.0)
    B = torch.from_numpy(wl.matrix_normal(n, nrhs, seed=n + 1).astype(np.float32)).cuda()
    piv = torch.arange(n, dtype=torch.int32, device="cuda")
    want = B.clone()
    api.lu_solve_f32(L, piv, want)
    torch.cuda.synchronize()
    g.set_wait_config(g.LU_WAIT_SITE_SOLVE, 50_000_000, 1)
    try:
        t0 = time.perf_counter()
        with pytest.raises(g.LuError) as exc:
            api.lu_solve_f32(L, piv, B.clone())
        dt = time.perf_counter() - t0
    finally:
        g.set_wait_config(g.LU_WAIT_SITE_SOLVE, 0, 0)
    assert exc.value.code == g.LU_ETIMEOUT
    assert 0.04 <= dt < 1.0, dt
    X = B.clone()
    api.lu_solve_f32(L, piv, X)
    assert torch.equal(X, want)

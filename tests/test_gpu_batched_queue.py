"""The queue of the batched factorization (csrc/batched.cu): every matrix is
taken once, from both ends, whatever the sizes."""
import numpy as np
import pytest

from tests.gpu_util import cuda_or_fail, lib

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype", ["f64", "f32"])
@pytest.mark.parametrize("count,big", [(1, 0), (305, 3), (3000, 0), (3000, 40)])
def test_every_matrix_is_factored_once(dtype, count, big):
    """Many tiny matrices, some large ones among them, sizes of nought and out
    of range: each equals the one factored in a call of its own."""
    torch = cuda_or_fail()
    g = lib()
    dt = torch.float64 if dtype == "f64" else torch.float32
    rng = np.random.default_rng(count + big)
    ns = rng.integers(1, 24, size=count)
    ns[rng.permutation(count)[:big]] = rng.integers(300, 700, size=big)
    t = torch.Generator(device="cuda")
    t.manual_seed(count)
    A0 = [torch.randn(int(n), int(n), generator=t, device="cuda", dtype=dt) for n in ns]
    As = [a.clone() for a in A0]
    pivs, info = g.lu_factor_batched(As)
    assert int(info.cpu().abs().max()) == 0
    for i in rng.permutation(count)[:25]:
        one = [A0[i].clone()]
        p, _ = g.lu_factor_batched(one)
        assert torch.equal(one[0], As[i]) and torch.equal(p[0], pivs[i])
    n = torch.from_numpy(ns).cuda()
    done = torch.stack([(a != a0).any() for a, a0 in zip(As, A0)])
    assert bool((done | (n == 1)).all())               # (a matrix of order 1 is its own factor)

"""The split residual (csrc/residual_split.cu) where its right-hand sides, or
A's rows, differ in their gradings: every element of R = B - A X is held to
n roundings of its own |A| |X| + |B|, and no element depends on which others
share its call."""
import numpy as np
import pytest

import workloads as wl
from tests.gpu_util import cuda_or_fail, lib
from tests.test_gpu_panel_edges import _exact_residual

pytestmark = pytest.mark.gpu


def _data(n, nrhs, kind):
    """A, X, B; within every 64 columns of A and rows of X lie all gradings."""
    A, X = wl.matrix_normal(n, n, seed=n + 5), wl.matrix_normal(n, nrhs, seed=n + 6)
    B = wl.matrix_normal(n, nrhs, seed=n + 7)
    k = np.arange(n)
    if kind.startswith("plain"):              # column 0 plain, the others graded against A
        w = int(kind[5:])
        d = (k * 7) % (2 * w) - w
        A = np.ldexp(A, d[None, :])
        X[:, 1:] = np.ldexp(X[:, 1:], -d[:, None])
    elif kind == "two ways":                  # one column against A, the next one with it
        d = (k * 7) % 80 - 40
        A = np.ldexp(A, d[None, :])
        X[:, ::2], X[:, 1::2] = np.ldexp(X[:, ::2], -d[:, None]), np.ldexp(X[:, 1::2], d[:, None])
    elif kind == "few":                       # a column's few entries meet A's smallest ones, another's the largest
        A[:, k % 8 != 0] *= 2.0 ** -55
        for c in range(1, nrhs):
            X[(k + c) % 8 != 0, c] = 0.0
    elif kind == "diagonal":                  # one large entry in a chunk, X's there of any size
        A = np.ldexp(A, -30)
        A[k, k] = 3.0
        X = np.ldexp(X, -((k[:, None] * 5 + 3 * np.arange(nrhs)[None, :]) % 40))
    return A, X, B


def _residual(A, X, B):
    torch = cuda_or_fail()
    g = lib()
    R, _ = g.lu_residual(torch.from_numpy(A.copy()).cuda(), torch.from_numpy(X.copy()).cuda(),
                         torch.from_numpy(B.copy()).cuda())
    return R.cpu().numpy()


@pytest.mark.parametrize("n,nrhs", [(256, 2), (256, 16), (333, 5), (400, 17)])
@pytest.mark.parametrize("kind", ["plain8", "plain10", "plain13", "plain20", "plain40", "two ways", "few", "diagonal"])
def test_each_column_within_its_own_bound(n, nrhs, kind):
    A, X, B = _data(n, nrhs, kind)
    err = np.abs(_residual(A, X, B) - _exact_residual(A, X, B))
    assert (err <= n * 2.0 ** -53 * (np.abs(A) @ np.abs(X) + np.abs(B))).all()


@pytest.mark.parametrize("kind", ["plain10", "plain40", "few", "diagonal"])
def test_a_column_is_the_same_alone_and_among_others(kind):
    A, X, B = _data(320, 16, kind)
    R = _residual(A, X, B)
    for c in (0, 1, 7, 15):
        np.testing.assert_array_equal(_residual(A, X[:, [c]], B[:, [c]])[:, 0], R[:, c])


@pytest.mark.parametrize("kind", ["plain10", "diagonal"])
def test_a_row_is_the_same_beside_other_rows(kind):
    A, X, B = _data(320, 4, kind)
    R = _residual(A, X, B)
    A2 = A.copy()
    A2[1::2] = np.ldexp(A2[1::2], (np.arange(320) * 11 % 90 - 45)[None, :])
    A2[3, 70], A2[5, 200] = np.inf, np.nan
    np.testing.assert_array_equal(_residual(A2, X, B)[::2], R[::2])


@pytest.mark.parametrize("n,nrhs", [(255, 16), (256, 1), (257, 17), (333, 16), (1000, 33), (2500, 64)])
@pytest.mark.parametrize("kind", ["normal", "plain10", "diagonal"])
def test_the_form_without_workspace_has_the_same_bits(n, nrhs, kind):
    """What a call returns does not depend on whether its workspace was to be
    had: lu_residual_noalloc has none.  One and several splits of the columns,
    a last split that is short, rows and columns off the tiles, unaligned rows."""
    torch = cuda_or_fail()
    lib()
    from paper_2010_05975_gb300 import _native as nat
    L = nat.library()
    A, X, B = (torch.from_numpy(M.copy()).cuda() for M in _data(n, nrhs, kind))
    out = []
    for fn in (L.lu_residual, L.lu_residual_noalloc):
        R = torch.full((n, nrhs), float("nan"), dtype=torch.float64, device="cuda")
        eta = torch.full((nrhs,), float("nan"), dtype=torch.float64, device="cuda")
        assert fn(n, nrhs, A.data_ptr(), n, X.data_ptr(), nrhs, B.data_ptr(), nrhs, R.data_ptr(), nrhs,
                  eta.data_ptr(), torch.cuda.current_stream().cuda_stream) == 0
        out.append((R.cpu().numpy(), eta.cpu().numpy()))
    np.testing.assert_array_equal(out[0][0].view(np.int64), out[1][0].view(np.int64))
    np.testing.assert_array_equal(out[0][1], out[1][1])


@pytest.mark.parametrize("nrhs,passes", [(8, 1), (16, 1), (17, 2)])
def test_profiled_bytes_are_those_of_the_path_taken(nrhs, passes):
    """A is read once per 16 right-hand sides, and once for its norm, which the
    same class counts; digits and partial sums are less than a third of it at
    n = 2048."""
    torch = cuda_or_fail()
    g = lib()
    n = 2048
    A = torch.randn(n, n, dtype=torch.float64, device="cuda")
    X = torch.randn(n, nrhs, dtype=torch.float64, device="cuda")
    g.prof_begin()
    g.lu_residual(A, X, torch.zeros_like(X))
    torch.cuda.synchronize()
    moved = g.prof_end()["residual"]["bytes"] - 8 * n * n
    assert 8 * n * n * passes <= moved < 8 * n * n * passes * 4 / 3

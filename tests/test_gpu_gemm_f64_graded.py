"""The FP64 update C -= A B from digit products where the large entries of a row do not meet those
of a column: entries graded inside rows and columns, mostly zeros, subnormals, and the digits
that make the dropped digit pairs largest.

Bound per entry, from the construction: a 32-deep chunk is off by less than 2^-50 sum |a b| (digits)
or 32 x 2^-53 = 2^-48 sum |a b| (FMA loop), and enters C with at most two roundings of values below
|C| + sum |a b|, 2^-52 of them; a result below the normal range rounds to 2^-1074.
"""
import numpy as np
import pytest

from test_gpu_gemm_f64 import _update

pytestmark = pytest.mark.gpu


def _matrices(M, N, K, kind):
    rng = np.random.default_rng([M, N, K, 7])
    A, B, C = rng.standard_normal((M, K)), rng.standard_normal((K, N)), rng.standard_normal((M, N))
    if kind == "graded":
        A *= 10.0 ** rng.uniform(-30, 30, A.shape)
        B *= 10.0 ** rng.uniform(-30, 30, B.shape)
        C[::2] = 0.0
    if kind == "apart":  # [1, 1e-20, ...] times [0, 1, ...] and the like
        for X, ax in ((A, 1), (B, 0)):
            big = rng.integers(0, K, X.shape[1 - ax])
            X *= 1e-20
            i = np.arange(X.shape[1 - ax])
            if ax == 1:
                X[i, big] = rng.standard_normal(len(i))
            else:
                X[big, i] = np.where(rng.random(len(i)) < 0.5, 0.0, 1e15)
        C[:] = 0.0
    if kind == "sparse":
        A[rng.random(A.shape) < 0.8] = 0.0
        B[rng.random(B.shape) < 0.8] = 0.0
    if kind == "subnormal":
        A[::2] *= 1e-310
        A[1::3, ::2] *= 1e-315
        B *= 1e100
        C[:] = 0.0
    if kind == "digits":  # every product of a dropped pair at its largest, of one sign
        x = (129 * 2 ** 54 - 256 * sum(2 ** (9 * i) for i in range(1, 6))) * 2.0 ** -61
        A[:], B[:], C[:] = x, x, 0.0
        A[1::2], B[:, 1::2] = -x, -x
    return A, B, C


@pytest.mark.parametrize("kind", ["normal", "graded", "apart", "sparse", "subnormal", "digits"])
@pytest.mark.parametrize("M,N,K", [(2, 2, 2), (64, 64, 32), (65, 63, 31), (130, 70, 17), (70, 66, 33), (96, 64, 100)])
def test_update_error_by_entry(M, N, K, kind):
    A, B, C = _matrices(M, N, K, kind)
    got = _update(A, B, C)
    L = np.longdouble
    ref = C.astype(L) - A.astype(L) @ B.astype(L)
    size = np.abs(A).astype(L) @ np.abs(B).astype(L)
    chunks = (K + 31) // 32
    bound = 2.0 ** -48 * size + chunks * 2.0 ** -52 * (np.abs(C) + size) + 2.0 ** -1074
    assert np.all(np.abs(got - ref) <= bound)


def test_a_small_entry_of_a_row_counts():
    A, B = np.array([[1.0, 1e-20]]), np.array([[0.0], [1.0]])
    assert _update(A, B, np.zeros((1, 1)))[0, 0] == -1e-20

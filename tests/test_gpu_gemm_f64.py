"""The FP64 update C -= A B from exact digit products, against extended precision.

Error bound per entry and 32-deep chunk, from the construction: two FP64 roundings of
values no larger than |C| + |A B| + rowmax colmax (2 x 2^-53 each), and the 64-bit sum of
the digit products cut at 2^-54 rowmax colmax (at most two units): together below
2^-51 (|C| + |C'| + rowmax colmax), rowmax / colmax the largest entries of the row of A and
the column of B.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _update(A, B, C):
    import torch

    from paper_1409_0297_gb300 import binding as bind

    (M, K), N = A.shape, B.shape[1]
    lda, ldb, ldc = M + 3, K + 1, M + 2

    def dev(X, ld):
        buf = np.zeros((X.shape[1], ld))
        buf[:, : X.shape[0]] = X.T
        return torch.from_numpy(buf).cuda()

    a, b, c = dev(A, lda), dev(B, ldb), dev(C, ldc)
    bind.sp_schur_update(0, M, N, K, a.data_ptr(), lda, 0, b.data_ptr(), ldb, 0, c.data_ptr(), ldc, 0, 1)
    torch.cuda.synchronize()
    out = c.cpu().numpy()
    assert not out[:, M:].any()  # the padding rows stay untouched
    return out[:, :M].T


def _matrices(M, N, K, kind):
    rng = np.random.default_rng([M, N, K])
    A, B, C = rng.standard_normal((M, K)), rng.standard_normal((K, N)), rng.standard_normal((M, N))
    if kind == "scaled":  # rows and columns of very different size, zeros, cancellation
        A *= 10.0 ** rng.integers(-30, 30, size=(M, 1))
        B *= 10.0 ** rng.integers(-30, 30, size=(1, N))
        A[rng.random(A.shape) < 0.3] = 0.0
        A[M // 2] = 0.0
        C = (A.astype(np.longdouble) @ B.astype(np.longdouble)).astype(np.float64)
    if kind == "extreme":  # every digit at its largest, of either sign
        A = np.where(rng.random(A.shape) < 0.5, 1.0, -1.0) * (2.0 - 2.0 ** -52)
        B = np.sign(A[0][:, None]) * np.ones((K, N)) * (2.0 - 2.0 ** -52)
    return A, B, C


@pytest.mark.parametrize("kind", ["normal", "scaled", "extreme"])
@pytest.mark.parametrize("M,N,K", [(1, 1, 1), (64, 64, 32), (65, 63, 31), (130, 70, 17), (40, 200, 16),
                                   (70, 66, 33), (96, 64, 100)])
def test_update_error(M, N, K, kind):
    A, B, C = _matrices(M, N, K, kind)
    got = _update(A, B, C)
    ref = C.astype(np.longdouble) - A.astype(np.longdouble) @ B.astype(np.longdouble)
    chunks = (K + 31) // 32
    rc = np.abs(A).max(axis=1)[:, None] * np.abs(B).max(axis=0)[None, :]
    # partial sums of several chunks: at most |C| + K rowmax colmax
    size = np.abs(C) + np.abs(ref).astype(np.float64) + (K if chunks > 1 else 1) * rc
    assert np.all(np.abs(got - ref).astype(np.float64) <= chunks * 2.0 ** -51 * size)


@pytest.mark.parametrize("value", [np.inf, -np.inf, np.nan, 1e-200, 1e200])
def test_update_outside_the_digit_range(value):
    """Infinities, NaNs and entries beyond the scales go through plain FMAs."""
    A, B, C = _matrices(70, 70, 20, "normal")
    A[3, 4] = value
    B[7, 66] = value
    got = _update(A, B, C)
    with np.errstate(all="ignore"):
        ref = C - A @ B
    fin = np.isfinite(ref)
    assert np.array_equal(np.isnan(got), np.isnan(ref))
    assert np.array_equal(got[~fin & ~np.isnan(ref)], ref[~fin & ~np.isnan(ref)])
    bound = 20 * 2.0 ** -52 * (np.abs(C) + np.abs(np.where(np.isfinite(A), A, 0)) @ np.abs(np.where(np.isfinite(B), B, 0)))
    assert np.all(np.abs(got - ref)[fin] <= bound[fin] + 1e-300)

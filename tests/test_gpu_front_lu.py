"""The factorisation of dense fronts (panels, interchanges, row-block solve, update, inverses of
the 32-wide diagonal blocks) against the same arithmetic on the CPU, bit for bit in FP32.

The CPU side is LU with partial pivoting on the k eliminated rows, in panels of 32 columns: the
pivot is the largest magnitude of the column, ties to the smallest position; multipliers are the
entry times the rounded reciprocal of the pivot; every update is one fused multiply-add, in the
order of the pivots; the trailing update subtracts the sum of its products.  Fused multiply-adds
come from error-free sums and rounding to odd (Boldo and Melquiond, "Emulation of a FMA and
correctly rounded sums: proved algorithms using rounding to odd", IEEE Trans. Comput. 57, 2008),
so nothing is left to a tolerance.  Entries are small integers, which tie in most columns.
"""
import ctypes

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

NB = 32


def _two_sum(a, b):
    s = a + b
    t = s - a
    return s, (a - (s - t)) + (b - t)


def _odd(s, e):
    """s + e, |e| at most half an ulp of s, rounded to odd."""
    i = s.view(np.int64)
    away = (e > 0) == (s > 0)
    fix = (e != 0) & ((i & 1) == 0)
    return np.where(fix, np.where(away, i + 1, i - 1), i).view(np.float64)


def _split(a):
    t = a * 134217729.0
    h = t - (t - a)
    return h, a - h


def fma(a, b, c):
    """a b + c rounded once, in the type of c."""
    T = np.result_type(c)
    a, b, c = np.broadcast_arrays(np.asarray(a, np.float64), np.asarray(b, np.float64), np.asarray(c, np.float64))
    if T == np.float32:
        s, e = _two_sum(a * b, c)  # the product of two FP32 numbers is exact
        return _odd(np.ascontiguousarray(s), e).astype(np.float32)
    u = a * b
    (ah, al), (bh, bl) = _split(a), _split(b)
    ul = ((ah * bh - u) + ah * bl + al * bh) + al * bl
    th, tl = _two_sum(c, ul)
    vh, vl = _two_sum(u, th)
    z, ze = _two_sum(tl, vl)
    return vh + _odd(np.ascontiguousarray(z), ze)


def reference(A, k, cols):
    """(factored columns 0 .. k - 1 and cols, pivots) of the front A."""
    T = A.dtype.type
    W = np.concatenate([A[:, :k], A[:, cols]], axis=1).astype(T)
    m, piv = A.shape[0], np.zeros(k, np.int32)
    for j0 in range(0, k, NB):
        e = min(j0 + NB, k)
        for j in range(j0, e):
            p = j + int(np.argmax(np.abs(W[j:k, j])))  # the first of the largest
            piv[j] = p
            W[[j, p]] = W[[p, j]]
            inv = T(1) / W[j, j]
            W[j + 1:, j] *= inv
            W[j + 1:, j + 1:e] = fma(-W[j + 1:, j:j + 1], W[j:j + 1, j + 1:e], W[j + 1:, j + 1:e])
        L = W[j0:e, j0:e]
        for l in range(e - j0 - 1):
            W[j0 + l + 1:e, e:] = fma(-L[l + 1:, l:l + 1], W[j0 + l:j0 + l + 1, e:], W[j0 + l + 1:e, e:])
        if T == np.float32:
            acc = np.zeros_like(W[e:, e:])
            for l in range(j0, e):
                acc = fma(W[e:, l:l + 1], W[l:l + 1, e:], acc)
            W[e:, e:] -= acc
        elif e < m:  # FP64: the products are exact up to the digit sums' error, so not bits
            W[e:, e:] = (W[e:, e:].astype(np.longdouble) -
                         W[e:, j0:e].astype(np.longdouble) @ W[j0:e, e:].astype(np.longdouble)).astype(T)
    for j0 in range(0, k, NB):
        e = min(j0 + NB, k)
        D, n = W[j0:e, j0:e].copy(), e - j0
        X, Y = np.eye(n, dtype=T), np.eye(n, dtype=T)
        for l in range(n):
            X[l + 1:] = fma(-D[l + 1:, l:l + 1], X[l:l + 1], X[l + 1:])
        if T == np.float32:
            for i in reversed(range(n)):
                for l in range(i + 1, n):
                    Y[i] = fma(-D[i, l], Y[l], Y[i])
                Y[i] = Y[i] / D[i, i]
        else:
            for l in reversed(range(n)):
                Y[l] = Y[l] / D[l, l]
                Y[:l] = fma(-D[:l, l:l + 1], Y[l:l + 1], Y[:l])
        W[j0:e, j0:e] = np.tril(X, -1) + np.triu(Y)
    return W, piv


def factor(fronts, k, grid=0, wait_ns=2 * 10 ** 9):
    """(factored fronts, pivots, row permutations, status) from the device."""
    import torch

    from paper_1409_0297_gb300 import binding as B

    fn = B.LIB.sp_test_front_lu
    fn.restype = ctypes.c_int
    fn.argtypes = [ctypes.c_int] * 5 + [ctypes.c_double, ctypes.c_longlong] + [ctypes.c_void_p] * 3 + \
        [ctypes.POINTER(ctypes.c_int)]
    nf, m = fronts.shape[:2]
    f = torch.from_numpy(np.ascontiguousarray(fronts.transpose(0, 2, 1))).cuda()
    piv = torch.zeros(nf, k, dtype=torch.int32, device="cuda")
    perm = torch.zeros_like(piv)
    prec = B.SP_PREC_FP32 if fronts.dtype == np.float32 else B.SP_PREC_FP64
    st = ctypes.c_int(-1)
    rc = fn(prec, m, k, nf, grid, 1e-14, wait_ns, f.data_ptr(), piv.data_ptr(), perm.data_ptr(), ctypes.byref(st))
    assert rc == B.SP_OK
    return f.cpu().numpy().transpose(0, 2, 1), piv.cpu().numpy(), perm.cpu().numpy(), st.value


def integers(T, m, k, nf, kind, seed):
    """Fronts of small integers; every leading block nonsingular through its heavy permutation."""
    rng = np.random.default_rng([m, k, seed])
    A = rng.integers(-2, 3, size=(nf, m, m)).astype(T)
    if kind == "sparse":
        A *= rng.random(A.shape) < 0.1
        for a in A:  # a permuted unit diagonal among the candidates
            a[rng.permutation(k), np.arange(k)] += 3
    return A


def check(A, k, got, piv, perm, which, cols):
    for f in which:
        ref, rp = reference(A[f], k, cols)
        assert np.array_equal(piv[f], rp)
        order = np.arange(k)
        for j in range(k):
            order[[j, rp[j]]] = order[[rp[j], j]]
        assert np.array_equal(perm[f], order)
        assert np.array_equal(np.concatenate([got[f][:, :k], got[f][:, cols]], axis=1), ref)


# rows of the panels: one warp, one CTA of each shape, clusters of 2 to 16 CTAs, the grid
SHAPES = [(20, 20, 3), (33, 25, 2), (70, 64, 2), (131, 96, 2), (250, 40, 2), (511, 33, 2), (1023, 32, 2),
          (1100, 33, 1), (2100, 40, 1), (4200, 33, 1)]


@pytest.mark.parametrize("kind", ["dense", "sparse"])
@pytest.mark.parametrize("m,k,nf", SHAPES)
def test_fp32_bits(m, k, nf, kind):
    A = integers(np.float32, m, k, nf, kind, 1)
    got, piv, perm, st = factor(A, k)
    assert st == 0
    cols = np.unique(np.linspace(k, m - 1, 12).astype(int)) if m > k else np.zeros(0, int)
    check(A, k, got, piv, perm, range(nf), cols)


def test_fp32_bits_of_many_tall_fronts():
    """More fronts than SMs with 513 to 768 rows: six rows to a thread."""
    A = integers(np.float32, 600, 33, 153, "dense", 2)
    got, piv, perm, st = factor(A, 33)
    assert st == 0
    check(A, 33, got, piv, perm, (0, 152), np.array([33, 300, 599]))


@pytest.mark.parametrize("m,k,nf", [(20, 20, 3), (50, 25, 2), (70, 32, 2), (250, 32, 2), (600, 32, 2), (600, 32, 80),
                                    (1100, 30, 1), (2100, 32, 1), (4200, 32, 1)])
def test_fp64_pivots_and_multipliers(m, k, nf):
    """One panel in FP64, bit for bit: pivots compared on all bits of the magnitudes (here equal in
    their leading 30), multipliers from the correctly rounded reciprocal."""
    rng = np.random.default_rng([m, nf])
    A = np.where(rng.random((nf, m, m)) < 0.5, 1.0, -1.0) * (1.0 + rng.integers(0, 9, (nf, m, m)) * 2.0 ** -33)
    got, piv, perm, st = factor(A, k)
    assert st == 0
    check(A, k, got, piv, perm, {0, nf - 1}, np.zeros(0, int))

"""The pseudospectral operator bit for bit: the transform's steps are a radix 2 (odd powers),
radices 4 and a radix 3, twiddles before the forward and behind the inverse butterflies, every
complex product (fma(a.x, b.x, -a.y b.y), fma(a.x, b.y, a.y b.x)), q and D / N rounded before they
enter a butterfly.  The CPU side runs the same operations with emulated fused multiply-adds; an
FP32 preconditioner turns one last bit of the operator into another residual at 1e-12, so a launch
shape may not change one.
"""
import math

import numpy as np
import pytest

from test_gpu_front_lu import fma

pytestmark = pytest.mark.gpu


def _cmul(a, b):
    return fma(a[0], b[0], -a[1] * b[1]), fma(a[0], b[1], a[1] * b[0])


def _radices(n):
    p = (n // 3 if n % 3 == 0 else n).bit_length() - 1
    return [2] * (p & 1) + [4] * (p // 2) + [3] * (n % 3 == 0)


def _butterfly(v, inv):
    add = lambda a, b: (a[0] + b[0], a[1] + b[1])
    sub = lambda a, b: (a[0] - b[0], a[1] - b[1])
    turn = (lambda a: (-a[1], a[0])) if inv else (lambda a: (a[1], -a[0]))
    if len(v) == 2:
        return [add(v[0], v[1]), sub(v[0], v[1])]
    if len(v) == 3:
        h3 = 0.86602540378443864676372317075294
        t1, t2 = add(v[1], v[2]), turn(sub(v[1], v[2]))
        m = tuple(fma(-0.5, t, a) for t, a in zip(t1, v[0]))
        return [add(v[0], t1), tuple(fma(h3, t, a) for t, a in zip(t2, m)),
                tuple(fma(-h3, t, a) for t, a in zip(t2, m))]
    s0, s1, s2 = add(v[0], v[2]), sub(v[0], v[2]), add(v[1], v[3])
    s3 = turn(sub(v[1], v[3]))
    return [add(s0, s2), add(s1, s3), sub(s0, s2), sub(s1, s3)]


def _lines(x, inv):
    """Transform of the last axis of the pair of arrays x."""
    n = x[0].shape[-1]
    ang = [2.0 * math.pi * t / n for t in range(n // 2)]
    c, s = np.array([math.cos(a) for a in ang]), np.array([-math.sin(a) for a in ang])
    w = np.concatenate([c, -c]), np.concatenate([s, -s])
    if inv:
        w = w[0], -w[1]
    x = [np.array(v) for v in x]
    steps, l = [], 1
    for r in _radices(n):
        steps.append((r, l))
        l *= r
    for r, l in (reversed(steps) if inv else steps):
        nb = n // r
        b = np.arange(nb)
        m = b % l
        far = [(b - m) * r + m + k * l for k in range(r)]
        near = [b + k * nb for k in range(r)]
        src, dst = (far, near) if inv else (near, far)
        v = [(x[0][..., i], x[1][..., i]) for i in src]
        if inv:
            v = _butterfly(v, inv)
        if l > 1:
            t = m * (nb // l)
            v = [v[0]] + [_cmul(v[k], (w[0][t * k], w[1][t * k])) for k in range(1, r)]
        if not inv:
            v = _butterfly(v, inv)
        for k in range(r):
            x[0][..., dst[k]], x[1][..., dst[k]] = v[k]
    return x


def _axis(x, axis, inv):
    y = _lines([np.moveaxis(v, axis, -1) for v in x], inv)
    return [np.moveaxis(v, -1, axis) for v in y]


def _operator(d, n, s, q, x, fused):
    """x + G (q x) with the symbol's 4 pi^2 k^2 - s fused by the host compiler or not."""
    k = np.arange(n)
    k = np.where(k < n // 2, k, k - n).astype(float)
    k2 = sum(np.square(a) for a in np.meshgrid(*([k] * d), indexing="ij"))
    four = 4.0 * math.pi * math.pi
    den = fma(four, k2, np.full(k2.shape, -s)) if fused else four * k2 - s
    Dn = 1.0 / den / float(n ** d)
    y = [x.real * q, x.imag * q]
    for a in range(d - 1, 0, -1):  # axis 0 of the flat index is the last array axis
        y = _axis(y, a, False)
    y = _axis(y, 0, False)
    y = _axis([v * Dn for v in y], 0, True)
    for a in range(1, d):
        y = _axis(y, a, True)
    return (y[0] + x.real) + 1j * (y[1] + x.imag)


@pytest.mark.parametrize("d,n,b", [(2, 4, 2), (2, 6, 3), (2, 8, 2), (2, 12, 3), (2, 16, 4), (2, 32, 4), (2, 48, 6),
                                   (2, 64, 4), (2, 96, 6), (2, 128, 8), (2, 256, 16), (2, 768, 24), (3, 4, 2),
                                   (3, 8, 2), (3, 16, 4), (3, 24, 3), (3, 32, 4)])
def test_operator_bits(d, n, b):
    import torch

    from paper_1409_0297_gb300 import binding as B

    s = 4 * np.pi ** 2 * 10.5
    rng = np.random.default_rng([d, n])
    shape = (n,) * d
    x = rng.standard_normal(shape) + 1j * rng.standard_normal(shape)
    q = rng.uniform(-1.0, 1.0, shape)
    S = B.Solver(d, n, b, s, prec=B.SP_PREC_FP32, restart=2, setup_route=1)
    S.factor(torch.from_numpy(q.ravel()).cuda())
    xd = torch.from_numpy(x.ravel()).cuda()
    w = torch.empty_like(xd)
    S.matvec(xd, w)
    S.close()
    got = w.cpu().numpy().reshape(shape)
    assert any(np.array_equal(got, _operator(d, n, s, q, x, fused)) for fused in (True, False))


@pytest.mark.parametrize("n,b,P", [(6, 3, 210), (4, 2, 40), (16, 4, 5)])
def test_lines_of_stacked_vectors(n, b, P):
    """Vectors of a group behind one another: a CTA's lines cross from one to the next (6^2: four
    lines a CTA, six a vector).  Every problem gives the bits of a context of its own."""
    import torch

    from paper_1409_0297_gb300 import binding as B

    rng = np.random.default_rng(n)
    s = 4 * np.pi ** 2 * (10.5 + np.arange(P) % 7)
    x = torch.from_numpy(rng.standard_normal(P * n * n) + 1j * rng.standard_normal(P * n * n)).cuda()
    S = B.Solver(2, n, b, list(s), prec=B.SP_PREC_FP32, restart=2, setup_route=1)
    w = torch.empty_like(x)
    S.green(x, w)
    S.close()
    for p in sorted({0, 1, 2, P // 2, P - 1}):
        S = B.Solver(2, n, b, s[p], prec=B.SP_PREC_FP32, restart=2, setup_route=1)
        one = torch.empty(n * n, dtype=torch.complex128, device="cuda")
        S.green(x[p * n * n:(p + 1) * n * n].clone(), one)
        S.close()
        assert torch.equal(w[p * n * n:(p + 1) * n * n], one)

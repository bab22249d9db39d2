"""The Gram-Schmidt products and norms bit for bit: each of min(304, ceil(N / 1024)) CTAs takes a
contiguous share, a thread every 256th entry of it in order (one fused multiply-add per real
product), then pairs of lanes 16, 8, 4, 2 and 1 apart, the eight warps in order, and the CTAs'
sums strided over one warp.  Fused multiply-adds on the CPU are the emulated ones of the fronts'
test; GMRES with an FP32 preconditioner turns a last bit of these sums into another residual at
1e-12, so a launch shape may not change one.
"""
import ctypes

import numpy as np
import pytest

from test_gpu_front_lu import fma

pytestmark = pytest.mark.gpu


def _tree(a):
    """Sum over the last axis of 32 lanes, lane i + lane i + 16, then 8, ..."""
    for o in (16, 8, 4, 2, 1):
        a = a[..., :o] + a[..., o:2 * o]
    return a[..., 0]


def _sum(N, step):
    """step(acc, i) adds the entries i to the accumulators of as many threads."""
    nblk = max(1, min(304, -(-N // 1024)))
    per = -(-N // nblk)
    part = np.zeros(nblk)
    t = np.arange(256)
    for c in range(nblk):
        c0, c1 = c * per, min(N, (c + 1) * per)
        acc = np.zeros(256)
        for g in range(c0, c1, 256):
            i = g + t
            live = i < c1
            acc[live] = step(acc[live], i[live])
        for s in _tree(acc.reshape(8, 32)):
            part[c] += s
    lanes = np.zeros(32)
    for g in range(0, nblk, 32):
        p = part[g:g + 32]
        lanes[:len(p)] += p
    return _tree(lanes)


@pytest.mark.parametrize("N,nv", [(1, 1), (255, 2), (1025, 8), (4096, 9), (9216, 3), (147456, 17), (350000, 2)])
def test_dots_and_norm(N, nv):
    import torch

    from paper_1409_0297_gb300 import binding as B

    fn = B.LIB.sp_test_dots
    fn.restype = ctypes.c_int
    fn.argtypes = [ctypes.c_longlong, ctypes.c_int] + [ctypes.c_void_p] * 4
    rng = np.random.default_rng([N, nv])
    V = rng.standard_normal((nv, N)) + 1j * rng.standard_normal((nv, N))
    w = rng.standard_normal(N) + 1j * rng.standard_normal(N)
    Vd, wd = torch.from_numpy(V).cuda(), torch.from_numpy(w).cuda()
    h = torch.zeros(nv, dtype=torch.complex128, device="cuda")
    nrm = torch.zeros(1, dtype=torch.float64, device="cuda")
    assert fn(N, nv, Vd.data_ptr(), wd.data_ptr(), h.data_ptr(), nrm.data_ptr()) == B.SP_OK
    got = h.cpu().numpy()
    for j in sorted({0, nv // 2, nv - 1}):
        v = V[j]
        re = _sum(N, lambda a, i: fma(v.real[i], w.real[i], fma(v.imag[i], w.imag[i], a)))
        im = _sum(N, lambda a, i: fma(v.real[i], w.imag[i], fma(-v.imag[i], w.real[i], a)))
        assert got[j] == re + 1j * im
    assert float(nrm) == np.sqrt(_sum(N, lambda a, i: fma(w.real[i], w.real[i], fma(w.imag[i], w.imag[i], a))))

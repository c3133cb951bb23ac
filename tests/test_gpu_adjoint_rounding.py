"""The adjoint's FP32 arithmetic, bit by bit: the order of the coefficient gradient's
sums and the input gradient's formulas, restated in numpy with exact fused
multiply-adds.  Training divides a nearly zero gradient by its own size (Adam's first
step), so another order of the same sums, as accurate as this one, changes the trained
coefficients visibly."""
import numpy as np
import pytest

import dpd_synth as synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_1612_09001_gb300 as dpd  # noqa: E402
from paper_1612_09001_gb300 import _lib  # noqa: E402

F32 = np.float32
WARPS, SUB, V = 12, 4, 4   # of the coefficient gradient: warps per CTA, units per warp and tile, samples per lane


def fma(a, b, c):
    """fl32(a b + c), rounded once: the product is exact in FP64, the sum is rounded to
    odd there (its error from a two-sum), which makes the rounding to FP32 the only one."""
    p, c = a.astype(np.float64) * b.astype(np.float64), np.asarray(c, np.float64)
    s = p + c
    z = s - p
    e = (p - (s - z)) + (c - z)
    bits = s.view(np.int64)
    odd = np.where((e != 0) & (bits & 1 == 0), np.where((e > 0) == (s > 0), bits + 1, bits - 1), bits)
    return odd.view(np.float64).astype(F32)


def _lane_sum(v):
    """Over the last axis (32 lanes): pairs 16 apart, then 8, 4, 2, 1."""
    for o in (16, 8, 4, 2, 1):
        v = v[..., :o] + v[..., o:2 * o]
    return v[..., 0]


def _gh(x, gy, P, Q, M, blocks):
    """One tap group of all M + 1 taps, `blocks` CTAs: [K] complex64."""
    Bp, Bq, T = (P + 1) // 2, (Q + 1) // 2, M + 1
    B, n, tile = max(Bp, Bq), len(x), WARPS * SUB * 32 * V
    tiles = -(-n // tile)
    rounds = -(-tiles // blocks)
    pad = lambda z: np.concatenate([z, np.zeros(rounds * blocks * tile + T - n, np.complex64)])
    xp, gp = pad(x), pad(gy)
    # sample of (CTA, warp, lane) in round i, unit j, position v
    at = (np.arange(blocks)[:, None, None] * tile + np.arange(WARPS)[:, None] * 32 * V + np.arange(32) * V)
    X, Y = (np.zeros((2, B, T) + at.shape, F32) for _ in range(2))
    c = np.zeros((2,) + at.shape, F32)
    for i in range(rounds):
        for j in range(SUB):
            s0 = at + i * blocks * tile + j * WARPS * 32 * V
            for v in range(V):
                c = c + np.stack([gp[s0 + v].real, gp[s0 + v].imag])
            for v in range(V):
                xr, xi = xp[s0 + v].real, xp[s0 + v].imag
                r = fma(xr, xr, xi * xi)
                p = np.stack([xr, xi])
                for b in range(B):
                    p = p * r if b else p
                    for k in range(T):
                        g = gp[s0 + v + k]
                        X[:, b, k] = fma(p, np.stack([g.real, g.imag]), X[:, b, k])
                        Y[:, b, k] = fma(p, np.stack([g.imag, g.real]), Y[:, b, k])

    def row(a):   # lanes, then warps in order
        a, q = _lane_sum(a), np.zeros(a.shape[:-2], F32)
        for w in range(WARPS):
            q = q + a[..., w]
        return q
    X, Y, c = row(X), row(Y), row(c)
    main = np.stack([X[0] + X[1], Y[0] - Y[1]])
    conj = np.stack([X[0] - X[1], Y[0] + Y[1]])
    rows = np.concatenate([main[:, :Bp].reshape(2, Bp * T, blocks), conj[:, :Bq].reshape(2, Bq * T, blocks),
                           c[:, None]], axis=1)
    re, im = rows.astype(np.float64).sum(axis=-1).astype(F32)
    return re + 1j * im


def _gx(x, gy, h, P, Q, M):
    """The Wirtinger form, tap by tap.  The coefficients' multiples by 1 .. B must be exact."""
    Bp, Bq, T, n = (P + 1) // 2, (Q + 1) // 2, M + 1, len(x)
    B = max(Bp, Bq)
    A, C = np.zeros((B + 1, T), np.complex64), np.zeros((B + 1, T), np.complex64)
    A[:Bp], C[:Bq] = h[:Bp * T].reshape(Bp, T), h[Bp * T:(Bp + Bq) * T].reshape(Bq, T)
    gp = np.concatenate([gy, np.zeros(T, np.complex64)])
    xr, xi = x.real, x.imag
    r, ur, ui = fma(xr, xr, xi * xi), fma(xr, xr, -xi * xi), F32(2) * xr * xi
    acc, ws = np.zeros((2, n), F32), np.zeros((2, n), F32)

    def chain(out, quads, g):
        a, b = (np.repeat(v[:, None], n, axis=1) for v in (quads[-1][:2], quads[-1][2:]))
        for q in quads[-2::-1]:
            a, b = fma(a, r, np.repeat(q[:2, None], n, 1)), fma(b, r, np.repeat(q[2:, None], n, 1))
        out = fma(a, np.stack([g.real, g.imag]), out)
        return fma(b, np.stack([g.imag, g.real]), out)
    quad = lambda e, f: np.array([e.real + f.real, e.real - f.real, e.imag + f.imag, f.imag - e.imag], F32)
    for k in range(T):
        g = gp[k:k + n]
        acc = chain(acc, [quad(F32(m + 1) * A[m, k], F32(m + 1) * C[m, k]) for m in range(B)], g)
        if B > 1:
            s = [np.array([C1.real + A1.real, C1.real - A1.real, C1.imag + A1.imag, A1.imag - C1.imag], F32)
                 for A1, C1 in ((F32(m + 1) * A[m + 1, k], F32(m + 1) * C[m + 1, k]) for m in range(B - 1))]
            ws = chain(ws, s, g)
    if B > 1:
        acc = fma(np.stack([ur, ur]), ws, acc)
        acc = fma(np.stack([-ui, ui]), ws[::-1], acc)
    return acc[0] + 1j * acc[1]


@pytest.mark.parametrize("P,Q,M", [(1, 0, 0), (1, 1, 1), (7, 7, 3), (7, 0, 3), (5, 3, 4), (11, 11, 2)])
@pytest.mark.parametrize("n", [1, 127, 6145, 3 * 6144, 7 * 6144 + 1001])
def test_gradients_to_the_bit(P, Q, M, n):
    x, gy = synth.clipped_gaussian(n, 0.3, key=(190, n)), synth.clipped_gaussian(n, 0.3, key=(191, n))
    h = synth.coeffs(P, Q, M, key=(192, P))
    h = (np.round(h.view(F32) * 2 ** 18) / 2 ** 18).astype(F32).view(np.complex64)
    f = dpd.DPD(P, Q, M)
    f.set_coeffs(h)
    blocks = min(3, -(-n // 1024))
    _lib.check("dpd_set_adj_launch", dpd.lib().dpd_set_adj_launch(f.handle, 3, M + 1))
    xd, gd = torch.from_numpy(x).cuda(), torch.from_numpy(gy).cuda()
    gh, gx = f.grad(xd, gd, gh=torch.empty(f.K, dtype=torch.complex64, device="cuda"), gx=torch.empty_like(xd))
    f.sync_status()
    f.close()
    assert np.array_equal(gh.cpu().numpy(), _gh(x, gy, P, Q, M, blocks))
    assert np.array_equal(gx.cpu().numpy(), _gx(x, gy, h, P, Q, M))

"""The pair factorisation and solves behind the least-squares estimates, at the
edges of their panels and row groups, and the problems left to the FP64 kernel."""
import numpy as np
import pytest

import dpd_synth as synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_1612_09001_gb300 as dpd  # noqa: E402


def _fit(P, Q, M, n, seed, precision="fp32"):
    """(h, G^{-1} g in FP64 from the library's own G and g): without refinement the
    estimate is the solve alone."""
    u = torch.from_numpy(synth.clipped_gaussian(n, 0.3, key=(140, seed))).cuda()
    h0 = synth.coeffs(P, Q, M, key=(141, seed))
    f = dpd.DPD(P, Q, M)
    f.set_coeffs(h0)
    t = f.apply(u)
    h, st = f.estimate(u, t, precision=precision, refine_iters=0)
    G, g, _ = f.gram(u, t, precision=precision)
    hb, info = f.estimate_batched([u] * 9, [t] * 9, precision=precision, refine_iters=0)
    f.close()
    assert info == [0] * 9
    G, g = G.cpu().numpy(), g.cpu().numpy()
    d = 1.0 / np.sqrt(np.real(np.diag(G)))
    A = G * d[:, None] * d[None, :]
    return h.cpu().numpy(), hb.cpu().numpy(), d * np.linalg.solve(A, d * g), np.linalg.cond(A), st


@pytest.mark.parametrize("P,Q,M", [(1, 0, 0), (1, 1, 1), (3, 0, 1), (5, 3, 0), (3, 3, 2), (7, 0, 7), (7, 7, 3), (5, 5, 5),
                                   (9, 0, 7), (7, 7, 7), (9, 9, 6), (11, 11, 7)])
def test_solve_at_panel_edges(P, Q, M):
    """K - 1 = 1 .. 96: part panels, whole panels, one row group and one past it.  The
    error of the solve is cond(A) times the factorisation's backward error, below
    2^-38 (element error 2^-42, at most 97 of them), and the FP32 rounding of h.  The
    nine problems of the batch sum their Gram matrix over fewer CTAs: the same result
    for each, within cond(A) times the FP32 Gram's 2e-6 of the single fit's."""
    h, hb, ref, cond, st = _fit(P, Q, M, 40000, P + 16 * M)
    err = np.linalg.norm(h - ref) / np.linalg.norm(ref)
    print(f"K {len(ref)} cond {cond:.2e} error {err:.2e} batch {np.linalg.norm(hb[0] - ref):.2e}")
    assert err <= cond * 2.0 ** -38 + 2.0 ** -23, (P, Q, M, cond)
    assert all(np.array_equal(hb[0], v) for v in hb[1:])
    assert np.linalg.norm(hb[0] - ref) <= (cond * 2e-6 + 2.0 ** -23) * np.linalg.norm(ref), (P, Q, M, cond)
    # the condition number is refined against G: Lanczos' 1e-11 and FP64 rounding on both sides
    print(f"cond error {abs(st['cond_est'] / cond - 1):.2e}")
    assert abs(st["cond_est"] - cond) <= (1e-10 + cond * 2.0 ** -48) * cond


def test_scales_at_the_edge_of_fp32():
    """Samples of 1e-16 (no constant in the target): Gram entries of 1e-29 to 1e-32
    beside the constant column's, split by their bits or through FP64 on either side of
    the limits, to the same coefficients."""
    n = 20000
    u0 = synth.clipped_gaussian(n, 0.3, key=(142, 0))
    f = dpd.DPD(1, 1, 3)
    h0 = synth.coeffs(1, 1, 3, key=(142, 1))
    h0[-1] = 0.0
    f.set_coeffs(h0)
    res = []
    for scale in (1.0, 1e-16):
        u = torch.from_numpy((u0 * np.float32(scale)).astype(np.complex64)).cuda()
        t = f.apply(u)
        h, _ = f.estimate(u, t, precision="fp32", refine_iters=2)
        res.append(h.cpu().numpy()[:-1])
    f.close()
    assert np.linalg.norm(res[0] - res[1]) <= 1e-4 * np.linalg.norm(res[0])


def test_collinear_columns_go_to_fp64():
    """A real-valued input makes the two branches' columns equal: pivots at rounding
    level, below the pair kernel's limit.  Whatever the FP64 kernel decides, the call
    returns as for any other fit (a status, or coefficients)."""
    n = 20000
    u = torch.from_numpy(np.abs(synth.clipped_gaussian(n, 0.3, key=(143, 0))).astype(np.complex64)).cuda()
    f = dpd.DPD(3, 3, 1)
    try:
        h, st = f.estimate(u, u, precision="fp32", refine_iters=0)
        assert h.numel() == f.K and st["cond_est"] > 1e6
    except dpd.DPDError as e:
        assert e.code == 6
    good = torch.from_numpy(synth.clipped_gaussian(n, 0.3, key=(143, 1))).cuda()
    hb, info = f.estimate_batched([good, u, good], [good, u, good], precision="fp32", refine_iters=0)
    assert info[0] == 0 and info[2] == 0
    e0 = np.zeros(f.K)
    e0[0] = 1.0
    assert np.abs(hb[0].cpu().numpy() - e0).max() <= 1e-3 and np.array_equal(hb[0].cpu().numpy(), hb[2].cpu().numpy())
    f.close()


def _nearly_real(n, seed):
    """Samples whose imaginary part is 2^-15 of their real part: the two branches' columns
    differ by that much, so the second branch's pivots are about 2^-28 times the first's
    (the difference is exact: both branches' Gram entries use the same real sums)."""
    a, b = synth.clipped_gaussian(n, 0.3, key=(144, seed)), synth.clipped_gaussian(n, 0.3, key=(145, seed))
    return torch.from_numpy((a.real + 1j * b.real * 2.0 ** -15).astype(np.complex64)).cuda()


@pytest.mark.parametrize("P,Q,M", [(1, 1, 0), (1, 1, 3), (3, 3, 3), (3, 3, 7), (5, 5, 5)])
@pytest.mark.parametrize("precision", ["fp32", "tf32x3"])
def test_fp64_factor_and_solve(P, Q, M, precision):
    """Smallest pivots between 1e-14 and 2^-25, which the pair kernel leaves to FP64:
    the coefficients against numpy's FP64 solve of the library's own G (its lower
    triangle, which the factorisation reads) and g, within K cond(A) 2^-53 and the FP32
    rounding of h, alone, as a batch of one (the same G) and beside problems that the pair
    kernel keeps."""
    n = 30000
    u = _nearly_real(n, M)
    f = dpd.DPD(P, Q, M)
    f.set_coeffs(synth.coeffs(P, Q, M, key=(146, P)))
    t = f.apply(u)
    h, _ = f.estimate(u, t, precision=precision, refine_iters=0)
    h1, info1 = f.estimate_batched([u], [t], precision=precision, refine_iters=0)
    G, g, _ = f.gram(u, t, precision=precision)
    G, g = G.cpu().numpy(), g.cpu().numpy()
    d = 1.0 / np.sqrt(np.real(np.diag(G)))
    A = np.tril(G) + np.tril(G, -1).conj().T
    A = A * d[:, None] * d[None, :]
    pivot, cond = np.abs(np.diag(np.linalg.cholesky(A))).min() ** 2, np.linalg.cond(A)
    assert 1e-14 < pivot < 2.0 ** -25, pivot
    ref = d * np.linalg.solve(A, d * g)
    for got in (h, h1[0]):
        err = np.linalg.norm(got.cpu().numpy() - ref) / np.linalg.norm(ref)
        print(f"K {f.K} pivot {pivot:.1e} cond {cond:.1e} error {err:.1e} = cond 2^{np.log2(err / cond):.1f}")
        assert err <= f.K * cond * 2.0 ** -53 + 2.0 ** -23
    assert info1 == [0]
    good = torch.from_numpy(synth.clipped_gaussian(n, 0.3, key=(147, 1))).cuda()
    tg = f.apply(good)
    hb, info = f.estimate_batched([good, u, good], [tg, t, tg], precision=precision, refine_iters=0)
    hg, _ = f.estimate_batched([good] * 3, [tg] * 3, precision=precision, refine_iters=0)
    assert info == [0, 0, 0] and torch.equal(hb[0], hg[0]) and torch.equal(hb[2], hg[0])
    f.set_coeffs(hb[1].contiguous())
    assert float((f.apply(u) - t).norm()) <= 1e-3 * float(t.norm())
    f.close()


@pytest.mark.parametrize("precision", ["fp32", "tf32x3", "bf16x3"])
def test_condition_of_the_factored_matrix(precision):
    """The condition number of the matrix that was factored (G's lower triangle) where the
    tensor-core forms leave the upper triangle 1e-10 off its conjugate: at 1e11 the two
    triangles' values differ by more than their sizes.  FP64 rounding of both sides is K
    2^-53 of the largest eigenvalue, so K cond 2^-53 relative, four times for the reference's."""
    u = _nearly_real(30000, 5)
    f = dpd.DPD(5, 5, 5)
    f.set_coeffs(synth.coeffs(5, 5, 5, key=(146, 5)))
    t = f.apply(u)
    _, st = f.estimate(u, t, precision=precision, refine_iters=0)
    G = f.gram(u, t, precision=precision)[0].cpu().numpy()
    f.close()
    d = 1.0 / np.sqrt(np.real(np.diag(G)))
    w = np.linalg.eigvalsh((np.tril(G) + np.tril(G, -1).conj().T) * d[:, None] * d[None, :])
    cond = w[-1] / w[0]
    print(f"cond {cond:.3e} error {abs(st['cond_est'] / cond - 1):.1e}")
    assert abs(st["cond_est"] / cond - 1) <= 1e-10 + 4 * len(d) * cond * 2.0 ** -53


@pytest.mark.parametrize("P,Q,M", [(1, 1, 1), (7, 7, 3), (9, 9, 6)])
@pytest.mark.parametrize("e", [-124, -120, -100, 100, 118, 121])
def test_targets_far_from_one(P, Q, M, e):
    """Targets scaled by 2^e, up to where their products with the basis still are FP32
    numbers: the solve of the library's own G and g within the bound of
    test_solve_at_panel_edges, in FP32's smallest and largest numbers too."""
    n = 400000
    u = torch.from_numpy(synth.clipped_gaussian(n, 0.3, key=(148, P))).cuda()
    f = dpd.DPD(P, Q, M)
    f.set_coeffs(synth.coeffs(P, Q, M, key=(149, P)))
    t = f.apply(u) * 2.0 ** e
    h, _ = f.estimate(u, t, precision="fp32", refine_iters=0)
    h1, _ = f.estimate_batched([u], [t], precision="fp32", refine_iters=0)
    G, g, _ = f.gram(u, t, precision="fp32")
    f.close()
    G, g = G.cpu().numpy(), g.cpu().numpy()
    d = 1.0 / np.sqrt(np.real(np.diag(G)))
    A = G * d[:, None] * d[None, :]
    ref, cond = d * np.linalg.solve(A, d * g), np.linalg.cond(A)
    assert np.all(np.isfinite(ref)) and np.abs(ref).max() < 1e38
    for got in (h, h1[0]):
        err = np.linalg.norm(got.cpu().numpy().astype(np.complex128) - ref) / np.linalg.norm(ref)
        # FP32's smallest step, 2^-149, is a rounding of its own for the coefficients themselves
        assert err <= cond * 2.0 ** -38 + 2.0 ** -23 + 2.0 ** -149 * len(ref) / np.linalg.norm(ref), (err, cond)


@pytest.mark.parametrize("nearly_real", [False, True])
def test_fit_without_statistics(nearly_real):
    """stats = NULL: the same coefficients (from either factorisation), and a Gram matrix
    that is not positive definite is still reported."""
    n = 20000
    u = _nearly_real(n, 3) if nearly_real else torch.from_numpy(synth.clipped_gaussian(n, 0.3, key=(150, 0))).cuda()
    f = dpd.DPD(3, 3, 3)
    f.set_coeffs(synth.coeffs(3, 3, 3, key=(151, 0)))
    t = f.apply(u)
    want, _ = f.estimate(u, t, refine_iters=1)
    h = torch.empty(f.K, dtype=torch.complex64, device="cuda")

    def call(x):
        return dpd.lib().dpd_estimate(f.handle, x.data_ptr(), t.data_ptr(), n, dpd.PRECISIONS["tf32x3"], 1, h.data_ptr(),
                                      None, torch.cuda.current_stream().cuda_stream)
    assert call(u) == 0 and torch.equal(h, want)
    assert call(torch.zeros_like(u)) == 6
    assert call(u) == 0 and torch.equal(h, want)
    f.close()

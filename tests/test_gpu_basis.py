"""The orthonormal basis of the least-squares estimates, formed on the device: at the
edges of its blocks of samples, per problem of a batch, and in the refinement's changes
of basis around the solve."""
import numpy as np
import pytest

import dpd_synth as synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_1612_09001_gb300 as dpd  # noqa: E402


@pytest.mark.parametrize("P,Q,M", [(1, 1, 2), (5, 3, 1), (0, 7, 1), (9, 9, 0), (11, 11, 1)])
@pytest.mark.parametrize("n", [300, 1024, 1025, 4097, 456 * 1024 + 3])
def test_orthogonal_estimate_over_lengths(P, Q, M, n):
    """A noiseless target in the model's range: the fit returns the generating
    coefficients through both bases of the solve; over a long record with a condition
    number that only an orthonormal basis has (the monomials' is 1e2 to 1e5 for the
    longer models; over a short one the branches are themselves correlated)."""
    u = torch.from_numpy(synth.clipped_gaussian(n, 0.3, key=(150, n))).cuda()
    h0 = synth.coeffs(P, Q, M, key=(151, P))
    f = dpd.DPD(P, Q, M)
    f.set_coeffs(h0)
    t = f.apply(u)
    h, st = f.estimate(u, t, precision="fp32", refine_iters=3, basis="orthogonal")
    hb, info = f.estimate_batched([u, u[: n // 2 * 2 - 64], u], [t, t[: n // 2 * 2 - 64], t], precision="fp32",
                                  refine_iters=3, basis="orthogonal")
    f.close()
    assert info == [0, 0, 0] and (n < 100000 or st["cond_est"] < 40.0)
    # The refined fit's own residual is the FP32 filter's rounding (6e-8 of t) and what the
    # rounding of h leaves: both far below 3e-6 of t.
    for got in (h.cpu().numpy(), hb[0].cpu().numpy(), hb[1].cpu().numpy(), hb[2].cpu().numpy()):
        psi = dpd.DPD(P, Q, M)
        psi.set_coeffs((got - h0).astype(np.complex64))
        e = psi.apply(u)
        psi.close()
        assert float(e.abs().square().sum() / t.abs().square().sum()) <= 1e-11

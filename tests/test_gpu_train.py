"""The kernels of a captured training step: the Adam update against FP64 numpy,
the loss's block sums at the edges of its blocks, and DirectLearner's route to
the Adam kernel."""
import numpy as np
import pytest

import dpd_synth as synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_1612_09001_gb300 as dpd  # noqa: E402
from paper_1612_09001_gb300 import _lib  # noqa: E402
from paper_1612_09001_gb300.direct import DirectLearner, SqErrorLoss, Transmitter  # noqa: E402


@pytest.mark.parametrize("n", [0, 1, 66, 255, 256, 257, 1000])
@pytest.mark.parametrize("t0", [0, 1, 6, 4095, 2.5])
def test_adam_step_against_fp64(n, t0):
    """One step from count t0 (2.5: not a whole number).  The FP64 result is rounded
    to FP32 once: half an ulp, doubled for the reference's own rounding."""
    rng = np.random.default_rng([n, int(10 * t0)])
    p, g, m = (rng.standard_normal(n).astype(np.float32) for _ in range(3))
    v = (rng.standard_normal(n) ** 2).astype(np.float32)
    if n:
        g[0] = v[0] = m[0] = 0.0   # 0 / (sqrt(0) + eps)
    lr, b1, b2, eps = np.float32(5e-3), 0.9, 0.999, 1e-8
    d = [torch.from_numpy(a.copy()).cuda() for a in (p, g, m, v)]
    step, dlr = torch.tensor(float(t0), device="cuda"), torch.tensor(float(lr), device="cuda")
    _lib.check("dpd_adam_step", dpd.lib().dpd_adam_step(*[a.data_ptr() for a in d], step.data_ptr(), n, dlr.data_ptr(),
                                                        b1, b2, eps, torch.cuda.current_stream().cuda_stream))
    t = t0 + 1.0
    g64 = g.astype(np.float64)
    m64 = b1 * m.astype(np.float64) + (1 - b1) * g64
    v64 = b2 * v.astype(np.float64) + (1 - b2) * g64 * g64
    p64 = p - float(lr) / (1 - b1 ** t) * m64 / (np.sqrt(v64 / (1 - b2 ** t)) + eps)
    assert float(step) == np.float32(t)
    for got, ref in zip((d[0], d[2], d[3]), (p64, m64, v64)):
        assert np.all(np.abs(got.cpu().numpy() - ref) <= 2.0 ** -23 * np.abs(ref) + 1e-44)


@pytest.mark.parametrize("n", [1, 31, 256, 257, 4 * 304 * 512, 4 * 304 * 512 + 1, 300007])
def test_sq_error_block_edges(n):
    y, x = synth.ofdm2(n, key=(131, n)), synth.ofdm2(n, key=(132, n))
    f = dpd.DPD(1, 0, 0)
    yd, xd = torch.from_numpy(y).cuda(), torch.from_numpy(x).cuda()
    gy = torch.empty_like(yd)
    e = y.astype(np.complex128) - (0.95 - 0.02j) * x.astype(np.complex128)
    for _ in range(2):   # the second call finds the completion counter cleared
        loss = f.sq_error(yd, xd, gain=0.95 - 0.02j, scale=0.5, gy=gy)
        ref = 0.5 * np.sum(np.abs(e) ** 2)
        assert abs(float(loss[0]) - ref) <= 1e-6 * ref
        assert np.abs(gy.cpu().numpy() - e).max() <= 1e-6 * np.abs(e).max()
    dl = torch.tensor(-1.75, device="cuda")   # the gradient alone, times dL
    _lib.check("dpd_sq_error_grad", dpd.lib().dpd_sq_error_grad(
        f.handle, yd.data_ptr(), xd.data_ptr(), n, 0.95, -0.02, 0.5, dl.data_ptr(), gy.data_ptr(),
        torch.cuda.current_stream().cuda_stream))
    assert np.abs(gy.cpu().numpy() + 1.75 * e).max() <= 1e-6 * np.abs(e).max()
    f.close()


@pytest.mark.parametrize("big", [3e19, float("inf")])
def test_sq_error_outside_fp32_sums(big):
    """Squares whose FP32 sum overflows are summed in FP64; an infinity stays one."""
    x = torch.zeros(800000, dtype=torch.complex64, device="cuda")   # four or more samples per thread
    y = torch.full_like(x, 1e19 if big != float("inf") else 1.0)
    y[::7777] = big if big == float("inf") else 1e19
    f = dpd.DPD(1, 0, 0)
    loss = float(f.sq_error(y, x, scale=1e-6 if big != float("inf") else 1.0)[0])
    if big == float("inf"):
        assert loss == float("inf")
    else:
        assert abs(loss - 8e37) <= 1e-5 * 8e37   # 8e5 samples of 1e38, scale 1e-6
    f.close()


def test_learner_steps_match_the_optimisers_own():
    """Steps through the Adam kernel against the same learner held to torch's Adam
    (a step hook keeps it there): the update is FP32-rounded in both, and eps = 1e-8
    turns a gradient's rounding into at most lr of a step for a coefficient whose
    gradient is itself rounding, so the trained coefficients agree to a fraction of lr."""
    t = synth.synthetic_pa(seed=1)
    x = torch.from_numpy(synth.ofdm2(1 << 14, key=(133, 0))).cuda()
    out = []
    for hooked in (False, True):
        lr = DirectLearner(x, Transmitter([t["iq"], t["pa"]]), 5, 5, 2, lr=5e-3)
        if hooked:
            lr.opt.register_step_post_hook(lambda *a: None)
        lr.capture()
        for _ in range(20):
            lr.step()
        torch.cuda.synchronize()
        out.append((lr.h.detach().clone(), float(lr.opt.state[lr.param]["step"])))
    assert out[0][1] == out[1][1] == 23.0
    assert float((out[0][0] - out[1][0]).abs().max()) <= 1e-4


def _loss_case(n=1000):
    x = torch.from_numpy(synth.ofdm2(n, key=(134, 0))).cuda()
    y0 = torch.from_numpy(synth.ofdm2(n, key=(135, 0))).cuda().requires_grad_()
    f = dpd.DPD(1, 0, 0)
    return x, y0, f, (2 * 0.25) * (y0 - (0.9 + 0.1j) * x).detach()


def test_loss_gradient_is_that_of_the_y_it_saw():
    x, y0, f, ref = _loss_case()
    y = y0 * 1
    loss = SqErrorLoss.apply(y, x, f, 0.9 + 0.1j, 0.25)
    with torch.no_grad():
        y.zero_()
    loss.backward()
    assert float((y0.grad - ref).abs().max()) <= 1e-6 * float(ref.abs().max())
    f.close()


def test_loss_gradient_is_differentiable_by_its_factor():
    x, y0, f, ref = _loss_case()
    loss = SqErrorLoss.apply(y0, x, f, 0.9 + 0.1j, 0.25)
    gl = torch.tensor(1.5, device="cuda", requires_grad=True)
    (gy,) = torch.autograd.grad(loss, y0, gl, create_graph=True)
    (d,) = torch.autograd.grad(torch.view_as_real(gy).square().sum(), gl)
    want = 2 * 1.5 * float(torch.view_as_real(ref).double().square().sum())
    assert abs(float(d) - want) <= 1e-5 * want
    f.close()


def test_loss_gradients_of_several_factors_at_once():
    x, y0, f, ref = _loss_case()
    loss = SqErrorLoss.apply(y0, x, f, 0.9 + 0.1j, 0.25)
    k = torch.tensor([1.0, -2.0, 0.5], device="cuda")
    (gy,) = torch.autograd.grad(loss, y0, k, is_grads_batched=True)
    assert float((gy - k[:, None] * ref).abs().max()) <= 2e-6 * float(ref.abs().max())
    f.close()


def test_learner_with_a_transmitter_of_its_own():
    """A callable that keeps its output and changes it after the loss."""
    x = torch.from_numpy(synth.ofdm2(4096, key=(136, 0))).cuda()
    kept = []

    def tx(v):
        kept.append(v * (1.1 + 0.1j))
        return kept[-1]
    lr = DirectLearner(x, tx, 3, 3, 1, lr=1e-3)
    want = DirectLearner(x, lambda v: v * (1.1 + 0.1j), 3, 3, 1, lr=1e-3)
    loss = lr.loss()
    with torch.no_grad():
        kept[-1].zero_()
    loss.backward()
    want.loss().backward()
    assert torch.equal(lr.param.grad, want.param.grad)


def test_adam_step_at_the_ends_of_fp32():
    """An infinite second moment (gradients above 2^64 overflow its FP32 storage) gives
    steps of zero, as sqrt(inf) does; infinite and NaN gradients give NaN."""
    inf, nan = float("inf"), float("nan")
    g = np.array([0.0, 1e25, 1e-30, inf, nan, 3e38], np.float32)
    m = np.array([1.0, 1e24, 0.0, 0.0, 0.0, 0.0], np.float32)
    v = np.array([inf, inf, 1e-45, 1.0, 1.0, 0.0], np.float32)
    p = np.ones(6, np.float32)
    d = [torch.from_numpy(a.copy()).cuda() for a in (p, g, m, v)]
    step, lr = torch.tensor(5.0, device="cuda"), torch.tensor(1e-2, device="cuda")
    _lib.check("dpd_adam_step", dpd.lib().dpd_adam_step(*[a.data_ptr() for a in d], step.data_ptr(), 6, lr.data_ptr(),
                                                        0.9, 0.999, 1e-8, torch.cuda.current_stream().cuda_stream))
    with np.errstate(all="ignore"):
        m64 = 0.9 * m.astype(np.float64) + (1 - 0.9) * g.astype(np.float64)
        v64 = 0.999 * v.astype(np.float64) + (1 - 0.999) * g.astype(np.float64) ** 2
        p64 = p - float(lr) / (1 - 0.9 ** 6) * m64 / (np.sqrt(v64 / (1 - 0.999 ** 6)) + 1e-8)
    got = d[0].cpu().numpy()
    assert np.array_equal(np.isnan(got), np.isnan(p64)) and np.allclose(got, p64, rtol=2.0 ** -23, atol=0, equal_nan=True), got

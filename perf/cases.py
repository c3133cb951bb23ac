"""Workloads of the predistortion library for performance measurement.

Each case is a call (or a short run of calls) that a program of a transmit
chain makes through the public entry points, on sizes that such a program
meets.  Kinds:

  apply           one block of samples through ``DPD.apply``
  stream          consecutive blocks of one transmit stream, ``DPD.apply_stream``
  host            samples in pinned host memory, ``DPD.apply_host`` (zero copy)
  batch           antenna streams of mixed models and lengths, ``BatchedPlan.execute``
  autograd        forward and backward of ``autograd.DPDFunction`` (both gradients)
  grad            both gradients through ``DPD.grad`` into the caller's buffers
  learn           one captured training step of ``direct.DirectLearner``
  estimate        one least-squares fit with its statistics, ``DPD.estimate``
  estimate_batch  independent fits, one per antenna, ``DPD.estimate_batched``
"""
import math
import random

import torch

import paper_1612_09001_gb300 as dpd
from paper_1612_09001_gb300.autograd import DPDFunction
from paper_1612_09001_gb300.direct import DirectLearner, Transmitter

LEARN_RATE = 5e-3
LEARN_WARMUP = 3   # eager steps that DirectLearner.capture() runs before the capture


# ------------------------------------------------------------------- the cases
def listed():
    return [
        # a short block, where the cost is the call itself: coefficients set once from the host
        dict(name="apply_short", kind="apply", n=1 << 16, P=5, Q=5, M=2, coeffs="host", signal="gauss"),
        # the paper's model (P = 5, Q = 3, five taps) near its 1e5-sample block, odd length,
        # coefficients that an estimate left on the device
        dict(name="apply_paper", kind="apply", n=100003, P=5, Q=3, M=4, coeffs="device", signal="gauss"),
        # a long record (16 M samples of a two-carrier OFDM signal), the filter's throughput
        dict(name="apply_long", kind="apply", n=1 << 24, P=9, Q=9, M=4, coeffs="host", signal="ofdm"),
        # a continuous transmitter: 1 ms subframes at 30.72 MHz, the history carried between them
        dict(name="stream_subframes", kind="stream", n=30720, blocks=16, P=7, Q=7, M=3, coeffs="device", signal="ofdm"),
        # a baseband process that keeps its samples in host memory
        dict(name="host_zero_copy", kind="host", n=1 << 22, P=7, Q=7, M=3, coeffs="host", signal="ofdm"),
        # 64 antennas with their own models and lengths, one launch
        dict(name="batch_64", kind="batch", streams=64, nmin=1 << 12, nmax=1 << 20, layout=0),
        # gradient-based training by a program's own loop: forward, then both gradients
        dict(name="autograd_1m", kind="autograd", n=1 << 20, P=7, Q=7, M=3, coeffs="device", signal="ofdm"),
        # the adjoint of a long record of odd length, into buffers that the program keeps
        dict(name="grad_long", kind="grad", n=(1 << 23) + 4097, P=9, Q=9, M=4, coeffs="host", signal="ofdm"),
        # one training step of direct learning (three filters, loss, three adjoints, Adam)
        dict(name="learn_1m", kind="learn", n=1 << 20, P=7, Q=7, M=3, signal="ofdm"),
        # one fit of the indirect learning loop on a captured block of odd length
        dict(name="estimate_ila", kind="estimate", n=262143, P=7, Q=7, M=3, precision="tf32x3", refine=2, basis="monomial"),
        # the largest model on a long record, in the statistically orthogonal basis
        dict(name="estimate_long", kind="estimate", n=1 << 22, P=11, Q=11, M=7, precision="bf16x3", refine=3,
             basis="orthogonal"),
        # 256 antennas, each with the largest model, with the call's default options
        dict(name="estimate_256", kind="estimate_batch", n=1 << 16, count=256, ragged=False, P=11, Q=11, M=7,
             precision="tf32x3", refine=2, basis="monomial"),
    ]


def _log_size(rng, lo, hi):
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng: random.Random):
    kind = rng.choice(["apply", "apply", "stream", "host", "batch", "autograd", "grad", "learn", "estimate", "estimate",
                       "estimate_batch"])
    P = rng.choice([1, 3, 5, 7, 9, 11])
    Q = rng.choice([P, P, max(1, P - 2), 0])
    M = rng.randint(0, 7)
    c = dict(kind=kind, P=P, Q=Q, M=M)
    if kind == "apply":
        c.update(n=_log_size(rng, 1 << 10, 1 << 23), coeffs=rng.choice(["host", "device"]), signal=rng.choice(["gauss", "ofdm"]))
    elif kind == "stream":
        c.update(n=_log_size(rng, 1 << 10, 1 << 18), blocks=rng.randint(4, 32), coeffs=rng.choice(["host", "device"]),
                 signal="ofdm")
    elif kind == "host":
        c.update(n=_log_size(rng, 1 << 14, 1 << 22), coeffs="host", signal="ofdm")
    elif kind == "batch":
        nmin = 1 << rng.randint(10, 14)
        c = dict(kind=kind, streams=rng.randint(4, 64), nmin=nmin, nmax=_log_size(rng, 2 * nmin, 1 << 20),
                 layout=rng.randrange(1 << 20))
    elif kind in ("autograd", "grad"):
        c.update(n=_log_size(rng, 1 << 12, 1 << 22), coeffs=rng.choice(["host", "device"]) if kind == "grad" else "device",
                 signal=rng.choice(["gauss", "ofdm"]))
    elif kind == "learn":
        c.update(n=_log_size(rng, 1 << 14, 1 << 20), P=rng.choice([3, 5, 7, 9]), M=rng.randint(0, 4), signal="ofdm")
        c["Q"] = c["P"]
    elif kind == "estimate":
        c.update(n=_log_size(rng, 1 << 15, 1 << 22), P=rng.choice([3, 5, 7, 9, 11]), M=rng.randint(0, 7),
                 precision=rng.choice(["tf32x3", "bf16x3"]), refine=rng.randint(2, 3), basis="orthogonal")
        c["Q"] = c["P"]
        if c["precision"] == "tf32x3" and c["P"] <= 7:
            c["basis"] = rng.choice(["monomial", "orthogonal"])
    else:
        c.update(n=_log_size(rng, 1 << 12, 1 << 16), count=rng.randint(4, 200), ragged=rng.random() < 0.5,
                 P=rng.choice([5, 7, 9, 11]), M=rng.randint(1, 7), precision=rng.choice(["tf32x3", "bf16x3"]), refine=2,
                 basis="orthogonal")
        c["Q"] = c["P"]
        if not c["ragged"]:
            c["n"] += c["n"] % 2   # rows of one tensor: every other row would start off a 16-byte boundary
    return c


# ---------------------------------------------------------------------- inputs
def _gen(*key):
    g = torch.Generator(device="cuda")
    g.manual_seed(random.Random(repr(key)).getrandbits(62))
    return g


def _normal(g, n):
    return torch.view_as_complex(torch.randn(n, 2, generator=g, device="cuda")).mul_(math.sqrt(0.5))


def _gauss(n, g, rms=0.3):
    """Complex Gaussian samples, magnitudes clipped at 1."""
    z = _normal(g, n) * rms
    return (z / z.abs().clamp(min=1.0)).to(torch.complex64).contiguous()


def _ofdm(n, g, rms=0.25):
    """Two OFDM carriers (1024-point IFFT, 600 QPSK subcarriers, 72-sample
    cyclic prefix) at +-0.3 of Nyquist."""
    nsym = -(-n // 1096)
    bins = torch.cat([torch.arange(1, 301), torch.arange(724, 1024)]).cuda()
    t = torch.arange(n, device="cuda", dtype=torch.float64)
    z = torch.zeros(n, dtype=torch.complex64, device="cuda")
    for shift in (0.3, -0.3):
        bits = torch.randint(0, 2, (nsym, 600, 2), generator=g, device="cuda").float() * 2 - 1
        spec = torch.zeros(nsym, 1024, dtype=torch.complex64, device="cuda")
        spec[:, bins] = torch.view_as_complex(bits)
        sym = torch.fft.ifft(spec, dim=1)
        a = torch.cat([sym[:, 1024 - 72:], sym], dim=1).reshape(-1)[:n]
        ph = torch.remainder(t * (0.5 * shift), 1.0) * (2 * math.pi)
        z += a * torch.polar(torch.ones_like(ph), ph).to(torch.complex64)
    return (z * (rms / z.abs().square().mean().sqrt())).contiguous()


def _signal(case, n, g):
    return _ofdm(n, g) if case.get("signal") == "ofdm" else _gauss(n, g)


def _branches(order):
    return (order + 1) // 2 if order > 0 else 0


def _num_coeffs(P, Q, M):
    return (_branches(P) + _branches(Q)) * (M + 1) + 1


def _coeffs(P, Q, M, *key):
    """h_{1,0} = 1, other main taps of standard deviation 1e-2 / p, conjugate
    taps 1e-3 / q, constant 1e-3 (1 + j); complex64 on the host."""
    r = random.Random(repr(key))
    h = []
    for orders, std in ((range(1, P + 1, 2) if P else (), 1e-2), (range(1, Q + 1, 2) if Q else (), 1e-3)):
        for p in orders:
            for _ in range(M + 1):
                h.append(complex(r.gauss(0, 1), r.gauss(0, 1)) * std / p / math.sqrt(2.0))
    if P:
        h[0] = 1.0
    h.append(1e-3 * (1 + 1j))
    return torch.tensor(h, dtype=torch.complex64)


def _models(case):
    """The streams (n, P, M) of a batch: part of the case, not of its inputs."""
    r = random.Random(case["layout"])
    return [(r.randint(case["nmin"], case["nmax"]), r.choice((5, 7, 9)), r.randint(2, 6)) for _ in range(case["streams"])]


def _transmitter_stages():
    """I/Q modulator (gain 1.02, phase 2 degrees, LO leakage) and a PA with memory (P = 7, M = 3)."""
    phi = math.radians(2.0)
    k1 = (1 + 1.02 * complex(math.cos(phi), -math.sin(phi))) / 2
    k2 = (1 - 1.02 * complex(math.cos(phi), math.sin(phi))) / 2
    pa = _coeffs(7, 0, 3, "pa")
    pa[0], pa[4], pa[8], pa[16] = 1.0, -0.1, 0.02, 0.0
    return [dict(P=1, Q=1, M=0, h=torch.tensor([k1, k2, 0.005], dtype=torch.complex64)), dict(P=7, Q=0, M=3, h=pa)]


def _fit_data(f, n, g, *key):
    """Basis input u and target t of a fit: t = Psi(u) theta plus noise 60 dB below it."""
    u = _gauss(n, g)
    f.set_coeffs(_coeffs(f.P, f.Q, f.M, *key).cuda())
    return u, f.apply(u) + _normal(g, n) * 0.3e-3


def _batch_lengths(case):
    return [case["n"] - (i % 64 if case["ragged"] else 0) for i in range(case["count"])]


def _inputs(case, seed):
    kind = case["kind"]
    g = _gen(seed, 1)
    key = ("h", seed)
    if kind == "batch":
        return [(_gauss(n, g), _coeffs(P, P, M, i, *key)) for i, (n, P, M) in enumerate(_models(case))]
    if kind in ("estimate", "estimate_batch"):
        lengths = [case["n"]] if kind == "estimate" else _batch_lengths(case)
        f = dpd.DPD(case["P"], case["Q"], case["M"])
        data = [_fit_data(f, n, g, i, *key) for i, n in enumerate(lengths)]
        torch.cuda.synchronize()
        f.close()
        us, ts = [d[0] for d in data], [d[1] for d in data]
        if kind == "estimate":
            return us[0], ts[0]
        return (us, ts) if case["ragged"] else (torch.stack(us), torch.stack(ts))
    h = _coeffs(case["P"], case["Q"], case["M"], *key)
    if kind == "stream":
        return _signal(case, case["n"] * case["blocks"], g), h
    x = _signal(case, case["n"], g)
    if kind in ("autograd", "grad"):
        return x, h, _signal(case, case["n"], g) * 1e-2
    return x, h


def prepare(case, seed):
    kind = case["kind"]
    st = dict(case=case)
    data = _inputs(case, seed)
    if kind == "batch":
        streams = []
        for (n, P, M), (x, h) in zip(_models(case), data):
            streams.append(dict(x=x, y=torch.empty_like(x), P=P, Q=P, M=M, h=h))
        st.update(streams=streams, plan=dpd.BatchedPlan(streams))
    elif kind == "learn":
        st.update(learner=DirectLearner(data[0], Transmitter(_transmitter_stages()), case["P"], case["Q"], case["M"],
                                        lr=LEARN_RATE).capture(LEARN_WARMUP))
    elif kind in ("estimate", "estimate_batch"):
        f = dpd.DPD(case["P"], case["Q"], case["M"])
        f.set_estimate_basis(case["basis"])
        st.update(f=f, u=data[0], t=data[1])
    else:
        f = dpd.DPD(case["P"], case["Q"], case["M"])
        x, h = data[0], data[1]
        h = h.cuda() if case["coeffs"] == "device" else h
        f.set_coeffs(h)
        st.update(f=f, x=x)
        if kind == "stream":
            st["x"] = [b.clone() for b in x.split(case["n"])]
            st["y"] = [torch.empty_like(b) for b in st["x"]]
        elif kind == "host":
            st["x"] = x.cpu().pin_memory()
            st["y"] = torch.empty_like(st["x"]).pin_memory()
        elif kind == "autograd":
            st.update(x=x.requires_grad_(), h=h.requires_grad_(), gy=data[2])
        elif kind == "grad":
            st.update(gy=data[2], gx=torch.empty_like(x), gh=torch.empty(f.K, dtype=torch.complex64, device="cuda"))
    return st


# ------------------------------------------------------------------------- run
def run(st):
    case = st["case"]
    kind = case["kind"]
    if kind == "apply":
        return st["f"].apply(st["x"])
    if kind == "stream":
        st["f"].reset_stream()
        return [st["f"].apply_stream(x, out=y) for x, y in zip(st["x"], st["y"])]
    if kind == "host":
        return st["f"].apply_host(st["x"], out=st["y"], zero_copy=True)
    if kind == "batch":
        st["plan"].execute()
        return [s["y"] for s in st["streams"]]
    if kind == "autograd":
        y = DPDFunction.apply(st["x"], st["h"], st["f"])
        gx, gh = torch.autograd.grad(y, (st["x"], st["h"]), st["gy"])
        return dict(y=y, gx=gx, gh=gh)
    if kind == "grad":
        gh, gx = st["f"].grad(st["x"], st["gy"], gh=st["gh"], gx=st["gx"])
        return dict(gh=gh, gx=gx)
    if kind == "learn":
        loss = st["learner"].step()
        return dict(loss=loss, gh=st["learner"].h_grad(), h=st["learner"].h)
    if kind == "estimate":
        h, stats = st["f"].estimate(st["u"], st["t"], precision=case["precision"], refine_iters=case["refine"])
        return dict(h=h, cond=stats["cond_est"], residual=stats["rel_residual"])
    h, _ = st["f"].estimate_batched(st["u"], st["t"], precision=case["precision"], refine_iters=case["refine"])
    return h


# ------------------------------------------------------------------------ work
def _filter_flops(P, Q, M, n):
    """Two flops per fused multiply-add of the widely-linear form: per sample and
    tap, four real polynomials of B coefficients."""
    B = max(_branches(P), _branches(Q))
    return 2.0 * n * 4 * B * (M + 1)


def _grad_flops(P, Q, M, n):
    """Coefficient gradient: four real products per (order, tap); input gradient:
    the derivative polynomials' 8 B - 4 per tap."""
    B, T = max(_branches(P), _branches(Q)), M + 1
    return 2.0 * n * (4 * B * T + (8 * B - 4) * T)


def _fit_flops(case, n):
    """Correlations of the 2 B + 2 real signals over the lags (the Gram matrix),
    then per refinement the filter and the coefficient gradient."""
    B, T = max(_branches(case["P"]), _branches(case["Q"])), case["M"] + 1
    one = 2.0 * n * 4 * B * T
    return 2.0 * n * (2 * B + 2) * (2 * B + 2) * T + case["refine"] * 2 * one


def work(case):
    kind = case["kind"]
    if kind == "batch":
        ms = _models(case)
        return dict(bytes=16.0 * sum(n for n, _, _ in ms), flops=sum(_filter_flops(P, P, M, n) for n, P, M in ms))
    P, Q, M, n = case["P"], case["Q"], case["M"], case["n"]
    if kind == "stream":
        n = n * case["blocks"]
    if kind in ("apply", "stream", "host"):
        return dict(bytes=16.0 * n, flops=_filter_flops(P, Q, M, n))
    if kind == "autograd":
        return dict(bytes=32.0 * n, flops=_filter_flops(P, Q, M, n) + _grad_flops(P, Q, M, n))
    if kind == "grad":
        return dict(bytes=24.0 * n, flops=_grad_flops(P, Q, M, n))
    if kind == "learn":
        tx = [(1, 1, 0), (7, 0, 3)]
        fwd = sum(_filter_flops(p, q, m, n) for p, q, m in [(P, Q, M)] + tx)
        B, T = max(_branches(P), _branches(Q)), M + 1
        back = 2.0 * n * (4 * B * T + 4 + 28 * 4)
        return dict(bytes=8.0 * n, flops=fwd + back)
    if kind == "estimate":
        return dict(bytes=16.0 * n, flops=_fit_flops(case, n))
    return dict(bytes=16.0 * sum(_batch_lengths(case)), flops=sum(_fit_flops(case, m) for m in _batch_lengths(case)))


def tolerance(case):
    """About four times the errors against 64 bits seen over the listed cases:
    1e-7 for the filter, 1.5e-7 for the gradients, 1.1e-6 for a step's loss;
    fits 2e-6 (long record, BF16 split), the batch of ill-conditioned monomial
    fits 1.5e-5."""
    kind = case["kind"]
    if kind in ("apply", "stream", "host", "batch"):
        return dict(rel=5e-7, max=5e-6)
    if kind in ("autograd", "grad"):
        return dict(rel=1e-6, max=1e-5)
    if kind == "learn":
        return dict(rel=5e-6, max=5e-5)
    if kind == "estimate_batch" and case["basis"] == "monomial":
        return dict(rel=1e-4, max=1e-3)
    return dict(rel=5e-5, max=5e-4)


# --------------------------------------------------------------- 64-bit results
def _delay(z, k):
    return z if k == 0 else torch.cat([z.new_zeros(k), z[:-k]]) if k < z.numel() else torch.zeros_like(z)


def _filter64(x, h, P, Q, M):
    """Eq. 1 in complex128 (differentiable)."""
    T, Bp, Bq = M + 1, _branches(P), _branches(Q)
    r = x.real.square() + x.imag.square()
    y = None
    for k in range(T):
        z = None
        for first, nb, base in ((0, Bp, x), (Bp * T, Bq, x.conj())):
            if nb:
                a = h[first + (nb - 1) * T + k]
                for b in range(nb - 2, -1, -1):
                    a = a * r + h[first + b * T + k]
                z = a * base if z is None else z + a * base
        z = _delay(z, k)
        y = z if y is None else y + z
    return y + h[-1]


def _psi64(u, P, Q, M, lo, hi, U=None):
    """Rows lo .. hi of the basis matrix (complex128), the orders mixed by U if given."""
    T = M + 1
    first = max(0, lo - M)
    v = u[first:hi].to(torch.complex128)
    r = v.real.square() + v.imag.square()
    cols = []
    for nb, base in ((_branches(P), v), (_branches(Q), v.conj())):
        mono = []
        z = base
        for _ in range(nb):
            mono.append(z)
            z = z * r
        for b in range(nb):
            c = mono[b] if U is None else sum(U[a][b] * mono[a] for a in range(b + 1))
            for k in range(T):
                d = torch.cat([c.new_zeros(k), c[:c.numel() - k]]) if k else c   # exact past the first M rows, or at the start
                cols.append(d[lo - first:])
    cols.append(torch.ones(hi - lo, dtype=torch.complex128, device=u.device))
    return torch.stack(cols, dim=1)


def _fit64(case, u, t, stats):
    P, Q, M, n = case["P"], case["Q"], case["M"], u.numel()
    U = None
    if case["basis"] == "orthogonal":
        r = u.to(torch.complex128).abs().square()
        B = max(_branches(P), _branches(Q))
        mu = [float(r.pow(k).mean()) for k in range(1, 2 * B)]
        A = torch.tensor([[mu[a + b] for b in range(B)] for a in range(B)], dtype=torch.float64)
        U = torch.linalg.inv(torch.linalg.cholesky(A)).T.contiguous().tolist()
    K = _num_coeffs(P, Q, M)
    G = torch.zeros(K, K, dtype=torch.complex128, device="cuda")
    g = torch.zeros(K, dtype=torch.complex128, device="cuda")
    step = 1 << 19
    t64 = t.to(torch.complex128)
    for lo in range(0, n, step):
        psi = _psi64(u, P, Q, M, lo, min(n, lo + step), U)
        G += psi.mH @ psi
        g += psi.mH @ t64[lo:lo + step]
    d = G.diagonal().real.rsqrt()
    A = G * d[:, None] * d[None, :]
    L = torch.linalg.cholesky(A)
    h = torch.cholesky_solve((g * d)[:, None], L)[:, 0] * d
    hm = h
    if U is not None:   # back to the monomials: h[a, k] = sum_{b >= a} U[a][b] h_U[b, k]
        hm = h.clone()
        T, at = M + 1, 0
        for nb in (_branches(P), _branches(Q)):
            blk = h[at:at + nb * T].reshape(nb, T)
            mix = torch.tensor([[U[a][b] if b >= a else 0.0 for b in range(nb)] for a in range(nb)], dtype=torch.complex128,
                               device="cuda")
            hm[at:at + nb * T] = (mix @ blk).reshape(-1)
            at += nb * T
    if not stats:
        return hm
    ev = torch.linalg.eigvalsh(A)
    err = t64 - _filter64(u.to(torch.complex128), hm, P, Q, M)
    return dict(h=hm, cond=float(ev[-1] / ev[0]), residual=float(err.abs().square().sum() / t64.abs().square().sum()))


def exact(case, seed):
    kind = case["kind"]
    data = _inputs(case, seed)
    c128 = torch.complex128
    if kind == "batch":
        return [_filter64(x.to(c128), h.cuda().to(c128), P, P, M) for (n, P, M), (x, h) in zip(_models(case), data)]
    if kind == "estimate":
        return _fit64(case, data[0], data[1], True)
    if kind == "estimate_batch":
        return torch.stack([_fit64(case, u, t, False) for u, t in zip(*data)])
    P, Q, M = case["P"], case["Q"], case["M"]
    if kind == "learn":
        x = data[0].to(c128)
        stages = [(s["P"], s["Q"], s["M"], s["h"].cuda().to(c128)) for s in _transmitter_stages()]
        h0 = torch.zeros(_num_coeffs(P, Q, M), dtype=c128, device="cuda")
        h0[0] = 1.0
        param = torch.nn.Parameter(torch.view_as_real(h0).clone())
        opt = torch.optim.Adam([param], lr=LEARN_RATE, eps=1e-8)
        for _ in range(LEARN_WARMUP + 1):
            opt.zero_grad()
            y = _filter64(x, torch.view_as_complex(param), P, Q, M)
            for p, q, m, hs in stages:
                y = _filter64(y, hs, p, q, m)
            loss = (y - x).abs().square().sum() / x.abs().square().sum()
            loss.backward()
            opt.step()
        return dict(loss=loss.detach(), gh=torch.view_as_complex(param.grad), h=torch.view_as_complex(param.detach()))
    x, h = data[0].to(c128), data[1].cuda().to(c128)
    if kind in ("autograd", "grad"):
        x.requires_grad_()
        h.requires_grad_()
        y = _filter64(x, h, P, Q, M)
        gx, gh = torch.autograd.grad(y, (x, h), data[2].to(c128))
        return dict(y=y.detach(), gx=gx, gh=gh) if kind == "autograd" else dict(gh=gh, gx=gx)
    y = _filter64(x, h, P, Q, M)
    if kind == "stream":
        return list(y.split(case["n"]))
    return y.cpu() if kind == "host" else y

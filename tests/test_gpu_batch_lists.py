"""Work lists of the batched plan: one run of items per CTA where a CTA fills an SM,
items dealt out in order otherwise; each stream equals the single-stream filter (whose
packed arithmetic per sample is the same) whatever the list, from fewer sub-blocks than
CTAs to streams cut over several CTAs, with odd lengths and empty streams among them."""
import numpy as np
import pytest

import dpd_synth as synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_1612_09001_gb300 as dpd  # noqa: E402

SHAPES = [(6, 16, 2, 0, 4), (6, 16, 4, 0, 8), (8, 16, 4, 0, 8), (4, 4, 3, 0, 0), (4, 1, 2, 0, 0)]


def _streams(lengths, seed):
    rng = np.random.default_rng(seed)
    out = []
    for i, n in enumerate(lengths):
        P, M = int(rng.choice([1, 3, 5, 7, 9])), int(rng.integers(0, 7))
        x = torch.from_numpy(synth.clipped_gaussian(max(n, 1), 0.3, key=(170, seed, i))[:n].copy()).cuda()
        out.append(dict(x=x, y=torch.full_like(x, float("nan")), P=P, Q=P, M=M, h=synth.coeffs(P, P, M, key=(171, i))))
    return out


@pytest.mark.parametrize("lengths", [[1], [0, 3071, 0, 3073], [100, 700000, 5, 12289], [12288 * 40 + 1] * 3,
                                     [4097 + 611 * i for i in range(40)], [1 << 20, 1, (1 << 21) + 7, 0, 99999]])
def test_lists_cover_every_sample_once(lengths):
    streams = _streams(lengths, len(lengths))
    ref = []
    for s in streams:
        f = dpd.DPD(s["P"], s["Q"], s["M"])
        f.set_coeffs(s["h"])
        ref.append(f.apply(s["x"]) if s["x"].numel() else s["x"])
        f.close()
    plan = dpd.BatchedPlan(streams)
    for shape in [None] + SHAPES:
        if shape:
            plan.set_launch(*shape)
        for s in streams:
            s["y"].fill_(float("nan"))
        plan.execute()
        plan.sync_status()
        for s, r in zip(streams, ref):
            assert torch.equal(s["y"], r), (shape, s["P"], s["M"], s["x"].numel())
    plan.close()

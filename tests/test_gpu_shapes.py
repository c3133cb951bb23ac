"""The default launch shapes of the forward filter on either side of the lines between
them: every shape evaluates a sample with the same operations in the same order, so the
outputs are those of a fixed shape bit for bit (itself checked against the oracle
elsewhere)."""
import pytest

import dpd_synth as synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_1612_09001_gb300 as dpd  # noqa: E402


@pytest.mark.parametrize("P,Q,M", [(1, 1, 0), (3, 3, 2), (5, 5, 3), (7, 5, 3), (9, 9, 4), (11, 11, 7)])
@pytest.mark.parametrize("coeffs", ["host", "device"])
def test_default_shapes_agree_with_a_fixed_one(P, Q, M, coeffs):
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    g = torch.Generator(device="cuda").manual_seed(160 + P)
    x = torch.view_as_complex(torch.randn(80000 * sms + 2, 2, generator=g, device="cuda")) * 0.2
    h = torch.from_numpy(synth.coeffs(P, Q, M, key=(160, P)))
    f, ref = dpd.DPD(P, Q, M), dpd.DPD(P, Q, M)
    ref.set_coeffs(h)
    ref.set_fwd_launch(V=4, warps=4, stages=2, mode=3)
    s = torch.cuda.Stream()
    for per in (3000, 8500, 24000, 80000):
        for n in (per * sms - 1, per * sms + 1):
            y0 = ref.apply(x[:n])
            if coeffs == "host":
                f.set_coeffs(h)
                y = f.apply(x[:n])
            else:   # under capture the tables stay on the device
                f.set_coeffs(h.cuda())
                y = torch.empty_like(y0)
                torch.cuda.synchronize()
                graph = torch.cuda.CUDAGraph()
                with torch.cuda.graph(graph, stream=s):
                    f.apply(x[:n], out=y)
                graph.replay()
            assert torch.equal(y, y0), (P, Q, M, coeffs, n)
    f.sync_status()
    f.close()
    ref.close()

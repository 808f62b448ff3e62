"""The detector on stored packets (detect_kernel): blocks queue the packets of several rows of slots
and trace them in batches of 32.  Each packet's event depends on the packet alone, so lists of any
length and density give the events of one long list, exactly; the tallies count them."""
import numpy as np
import pytest

import mcv_inputs as mi

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

_FIELDS = ("x", "y", "z", "vx", "vy", "vz", "t", "w", "id", "order")


def _take(api, pk, index):
    out = api.NeutronBuffers(int(index.numel()), pk.fp_mode)
    for f in _FIELDS:
        setattr(out, f, getattr(pk, f)[index].contiguous())
    return out


@pytest.mark.parametrize("fp", ["FP32", "FP64"])
def test_events_do_not_depend_on_the_list(fp):
    from paper_1504_02776_gb300 import api, binding as B
    import gpu_helpers as H
    ctx = H.ctx()
    wl = mi.config2(n=60_000).replace(detector=mi.tube_detector(n_tof=40))
    pk = ctx.trace_packets(wl, fp_mode=getattr(B, fp))
    _, _, want = ctx.detect(wl, pk)
    filled = torch.nonzero(pk.order >= 0).flatten()
    real = torch.nonzero(pk.order >= 1).flatten()
    gen = torch.Generator(device="cuda").manual_seed(1)
    mixed = torch.randperm(pk.n, device="cuda", generator=gen)
    lists = [real[:n] for n in (1, 31, 32, 33, 127, 128, 129, 4099)]
    lists += [real, filled[:515], torch.cat([real[:700], filled[:90], real[700:1500]])]
    lists += [mixed[:n] for n in (511, 513, 40_001, 160_003)]
    for index in lists:
        q = _take(api, pk, index)
        counts, tallies, got = ctx.detect(wl, q)
        order = q.order.cpu().numpy()
        used = torch.from_numpy(order >= 0).to("cuda")
        for f in ("bin", "pixel", "tof", "w_det"):
            assert torch.equal(got[f][used], want[f][index][used]), (f, index.numel())
        real_bins = got["bin"].cpu().numpy()[order >= 1]
        beam, w_det, _, n_det, n_over, n_miss, _, n_emit = tallies.cpu().numpy()
        assert n_emit == real_bins.size and n_det == (real_bins >= 0).sum()
        assert n_over == (real_bins == -2).sum() and n_miss == (real_bins == -1).sum()
        total = got["w_det"].cpu().numpy()[order >= 1][real_bins >= 0].sum()
        assert np.isclose(counts.sum().item(), total, rtol=1e-12)
        # the tally's sums are compensated FP32 pairs in the FP32 mode
        assert np.isclose(w_det, total, rtol=1e-9)
        assert np.isclose(beam, q.w.double().cpu().numpy()[order == 0].sum(), rtol=1e-9)
    ctx.close()

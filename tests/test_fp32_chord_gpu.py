"""FP32 runs in a batch against the same simulations alone.  The kernels evaluate r^2 - d^2 of a tube
chord in one of two forms, each within 4 units of 2^-24 r^2, so a chord's weight, proportional to
its root, differs by up to 4 u r^2 / (r^2 - d^2) of itself.  Over impact parameters spread evenly
across the tube that is 4 u = 2.4e-7 of the summed weight, and the bar is four times that; a
packet is detected by one form and not by the other only within 8 u of the edge (1 in 4e6)."""
import pytest

import mcv_inputs as mi

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("make", [lambda n: mi.config2(n=n), lambda n: mi.powder_in_can(n=n),
                                  lambda n: mi.vanadium_powder(n=n),
                                  lambda n: mi.config3(n=n, rot_deg=30.0)],
                         ids=["powder", "can", "phonon", "crystal"])
def test_batch_and_single_runs_differ_by_their_chords_only(make):
    from paper_1504_02776_gb300 import binding as B
    import gpu_helpers as H
    ctx = H.ctx()
    wl = make(200_000).replace(detector=mi.tube_detector(n_tof=40))
    h, t = ctx.trace(wl, fp_mode=B.FP32)
    b = ctx.batch([wl], fp_mode=B.FP32)
    b.run(sync=True)
    hb, tb = b.hists[0]
    assert (hb - h).abs().sum().item() <= 1e-6 * h.sum().item()
    assert abs((tb[3] - t[3]).item()) <= 1 + t[3].item() * 1e-5
    b.close()
    ctx.close()

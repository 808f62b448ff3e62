"""The FP64 single-crystal kernel's root search (FP32 signs of the leading minors, FP64 where
they are not certain, a bracketed secant iteration) against the oracle's 33 nodes and 50
bisection steps, away from the benchmark's energy: slow neutrons (few roots, small Ef), the
upper end of the sweep (large phases, most roots), axis-parallel and general orientations.
Bars: the FP64 per-packet bars of the parity tests."""
import numpy as np
import pytest

import mcv_inputs as mi

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("ei,rot", [(12.0, 0.0), (30.0, 90.0), (120.0, 45.0), (500.0, 77.0)])
def test_fp64_crystal_roots_match_oracle(ei, rot):
    import oracle
    from paper_1504_02776_gb300 import binding as B
    import gpu_helpers as H
    ctx = H.ctx()
    wl = mi.config3(rot_deg=rot, n=1500)
    wl = wl.replace(beam=mi.powder_beam(ei=ei))
    pk, g = H.packets(ctx, wl, B.FP64)
    op = oracle.trace(wl, packets=True)["packets"]
    dev, bad = H.check_fp64_packets(g, op)
    assert not any(bad.values()), (bad, {f: float(d.max()) for f, d in dev.items()})
    assert np.count_nonzero(op["order"] >= 1) > 100
    ctx.close()

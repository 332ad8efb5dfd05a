"""The automatic layout of FP64 calls on mechanisms of few reactions: beyond the
line that the mechanism's size draws, the lane layout's result (its bits), before
it the warp layout's."""
import dataclasses

import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

from paper_1309_2710_gb300 import kin, synth  # noqa: E402


@pytest.mark.parametrize("nS,nR,method,energy,warp,lane", [
    (17, 20, kin.RKC, 0, 300, 360), (24, 60, kin.RKC, 0, 380, 420), (5, 8, kin.RKC, 1, 60, 70),
    (10, 12, kin.RKC, 1, 800, 900), (14, 20, kin.RKCK, 1, 240, 280), (9, 38, kin.RKCK, 1, 1000, None),
    (24, 100, kin.RKC, 1, 1000, None)])
def test_lines(nS, nR, method, energy, warp, lane):
    m = synth.make_mechanism(nS, nR, ("H", "O", "C", "N"), 0.1, 0.0, seed=nS + nR)
    if energy:
        cp, Hf = synth.make_thermo(m, 7)
        m = dataclasses.replace(m, cp=cp, Hf=Hf)
    sm = torch.cuda.get_device_properties(0).multi_processor_count
    km = kin.Mechanism(m)
    for per_sm, want in ((warp, kin.LAYOUT_WARP), (lane, kin.LAYOUT_LANE)):
        if per_sm is None:
            continue
        state = [torch.as_tensor(a).cuda() for a in synth.make_states(m, per_sm * sm, T_range=(900.0, 2000.0), seed=3)]
        got = {}
        for layout in (kin.LAYOUT_AUTO, kin.LAYOUT_WARP, kin.LAYOUT_LANE):
            T, p, Y = (a.clone() for a in state)
            kin.integrate(km, T, p, Y, 1e-9, 1e-6, 1e-10, method, sigma=kin.SIGMA_POWER, energy=energy, layout=layout)
            got[layout] = Y.cpu().numpy()
        other = kin.LAYOUT_WARP + kin.LAYOUT_LANE - want
        assert not np.array_equal(got[want], got[other])
        assert np.array_equal(got[kin.LAYOUT_AUTO], got[want])
    km.close()

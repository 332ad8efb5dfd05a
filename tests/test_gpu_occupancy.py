"""KIN_OCC_HIGH in the FP64 warp layout: the default budget's kernels unless the
call names more blocks per SM than they leave room for (10 and 6 of 128 threads are
the small budgets' most), and the same bits either way."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

from paper_1309_2710_gb300 import kin, synth  # noqa: E402


@pytest.mark.parametrize("wl,most", [("h2co_13sp_rkc", 10), ("ch4_53sp_rkc_mixed", 10), ("h2co_13sp_rkc_energy", 6),
                                     ((16, 250), 10), ((32, 250), 10)])
def test_budgets(wl, most):
    if isinstance(wl, str):
        m = synth.workload_mechanism(wl)
        state = synth.workload_states(wl, m, cells=700)
    else:
        m = synth.make_mechanism(*wl, ("H", "O", "C", "N"), 0.1, 0.04, seed=1)
        state = synth.make_states(m, 700, T_range=(900.0, 2000.0), seed=2)
    en = int(m.cp is not None)
    T, p, Y = (torch.as_tensor(a).cuda() for a in state)
    km = kin.Mechanism(m)
    ref = None
    for kw in (dict(), dict(occupancy=kin.OCC_HIGH), dict(occupancy=kin.OCC_HIGH, blocks_per_sm=2),
               dict(occupancy=kin.OCC_HIGH, blocks_per_sm=most)):
        y, t = Y.clone(), T.clone()
        sta = torch.zeros((700, kin.NSTATS), dtype=torch.int32, device="cuda")
        kin.integrate(km, t, p, y, 1e-8, 1e-6, 1e-10, kin.RKC, stats=sta, sigma=kin.SIGMA_POWER, energy=en,
                      layout=kin.LAYOUT_WARP, block_threads=128, **kw)
        got = [a.cpu().numpy() for a in (y, t, sta)]
        ref = ref or got
        assert (got[2][:, 1] > 0).all() and np.isfinite(got[0]).all()
        assert all(np.array_equal(a, b) for a, b in zip(got, ref)), kw
    km.close()

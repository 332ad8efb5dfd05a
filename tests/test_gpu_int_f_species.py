"""Rates of trace species in the FP64 kernels: kin.rates on unburnt mixtures within
the bounds of test_int_f_species.py, and one Cash-Karp step (so short that each
species moves by dt times its rate) in every layout, per species against the
oracle: 1e-11 of |Y| + dt sum_j |nu_ij Omega_j|, a hundred times the rates' bound."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

import oracle  # noqa: E402
from paper_1309_2710_gb300 import kin, synth  # noqa: E402
from tests import int_f_replay  # noqa: E402
from tests.test_int_f_species import RADICALS, ULP, unburnt  # noqa: E402

WORKLOADS = ["h2_9sp_rkck", "h2co_13sp_rkc", "ch4_53sp_rkc_mixed", "c2h4_111sp_rkc_batched"]


def dev(a):
    return torch.as_tensor(np.ascontiguousarray(a), device="cuda")


@pytest.mark.parametrize("radicals", RADICALS)
@pytest.mark.parametrize("wl", WORKLOADS)
def test_rates(wl, radicals):
    m = synth.workload_mechanism(wl)
    f = int_f_replay.Mech(None, m)
    T, p, Y = unburnt(wl, m, 12, radicals)
    km = kin.Mechanism(m)
    out = kin.rates(km, dev(T), dev(p), dev(Y), kin.FP64).cpu().numpy()
    km.close()
    for c in range(12):
        ref, mag = f.reference(T[c], p[c], Y[:, c])
        bound = ULP * (16 + 4 * (abs(m.lnA) + abs(m.beta) * np.log(T[c]) + m.Ea / (synth.R_GAS * T[c])).max())
        assert (np.abs(out[:, c] - ref) <= bound * mag).all(), c


@pytest.mark.parametrize("wl", WORKLOADS)
def test_one_step(wl):
    m = synth.workload_mechanism(wl)
    f = int_f_replay.Mech(None, m)
    n, dt = 12, 1e-13
    T, p, Y = unburnt(wl, m, n, (-24, -9))
    Yo, so, xo, _ = oracle.integrate(oracle.Mech(m), T, p, Y, dt, 1e-6, 1e-10, oracle.RKCK)
    mag = np.stack([f.reference(T[c], p[c], Y[:, c])[1] for c in range(n)], 1).astype(np.float64)
    km = kin.Mechanism(m)
    sm = torch.cuda.get_device_properties(0).multi_processor_count
    # (copies of the cells, options): warp layout with a whole and with half a warp per
    # cell, and the lane layout
    shapes = [(1, dict(layout=kin.LAYOUT_WARP)), (sm, dict(layout=kin.LAYOUT_WARP)),
              (900, dict(block_threads=128, blocks_per_sm=4) if m.n_species <= 16 else dict(layout=kin.LAYOUT_LANE))]
    for k, kw in shapes:
        Yd = dev(np.tile(Y, (1, k)))
        sta = torch.zeros((n * k, kin.NSTATS), dtype=torch.int32, device="cuda")
        kin.integrate(km, dev(np.tile(T, k)), dev(np.tile(p, k)), Yd, dt, 1e-6, 1e-10, kin.RKCK, stats=sta, **kw)
        Yg = Yd.cpu().numpy()
        assert np.array_equal(Yg, np.tile(Yg[:, :n], (1, k)))
        assert np.array_equal(sta.cpu().numpy()[:n], xo) and (xo[:, 1] == 1).all()
        err = np.abs(Yg[:, :n] - Yo) / (np.abs(Yo) + dt * mag)
        assert err.max() <= 1e-11, (k, kw, err.max())
    km.close()

"""The paths that the automatic choices take, against the oracle: the headline
workload's call (the lane layout's integer f), and the energy equation in the warp
layout with a whole, half and a quarter warp per cell (RKC) or a whole and half
(RKCK), with the same bits for each, and at the sizes where its lanes per cell and
vector slots change."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

import oracle  # noqa: E402
from paper_1309_2710_gb300 import kin, synth  # noqa: E402
from tests.oracle_variants import reference  # noqa: E402
from tests.parity import compare  # noqa: E402
from tests.test_gpu_int_f import Mech, dev  # noqa: E402


def run(km, T, p, Y, dt, method, **kw):
    n = T.size
    Td, Yd = dev(T), dev(Y)
    st = torch.full((n,), 255, dtype=torch.uint8, device="cuda")
    sta = torch.zeros((n, kin.NSTATS), dtype=torch.int32, device="cuda")
    kin.integrate(km, Td, dev(p), Yd, dt, 1e-6, 1e-10, method, status=st, stats=sta, max_steps=20000, **kw)
    return [a.cpu().numpy() for a in (Yd, Td, st, sta)]


def test_headline_call_sampled():
    name = "h2co_13sp_rkc"
    m = synth.workload_mechanism(name)
    T, p, Y = synth.workload_states(name, m)
    km = kin.Mechanism(m)
    Yg, _, stg, stag = run(km, T, p, Y, 1e-6, kin.RKC, sigma=kin.SIGMA_GERSHGORIN)
    km.close()
    at = np.sort(np.random.default_rng(19).choice(T.size, 768, replace=False))
    Yo, sto, stao, floor = reference(m, T[at], p[at], Y[:, at], 1e-6, 1e-6, 1e-10, oracle.RKC)
    compare(Yg[:, at], Yo, stg[at], sto, stag[at], stao, 1e-10, 1e-6, floor=floor)
    assert (stg == 0).all() and np.abs(Yg.sum(0) - 1).max() < 1e-12


@pytest.mark.parametrize("name", ["h2co_13sp_rkc_energy", "h2_9sp_rkck_energy"])
def test_energy_lanes(name):
    w = synth.WORKLOADS[name]
    m = synth.workload_mechanism(name)
    T, p, Y = synth.workload_states(name, m, cells=48, seed_offset=71)
    sm = torch.cuda.get_device_properties(0).multi_processor_count
    km = kin.Mechanism(m)
    ref = None
    for per_sm in (0, 9, 80):  # RKC: a whole, half and a quarter warp per cell
        k = max(1, per_sm * sm // 48 + 1 if per_sm else 1)
        got = run(km, np.tile(T, k), np.tile(p, k), np.tile(Y, (1, k)), w["dt"], w["method"], sigma=kin.SIGMA_POWER,
                  energy=1)
        assert all(np.array_equal(a, np.concatenate([a[..., :48]] * k, -1)) for a in (got[0], got[1], got[2], got[3].T))
        got = [got[0][:, :48], got[1][:48], got[2][:48], got[3][:48]]
        ref = ref or got
        assert all(np.array_equal(a, b) for a, b in zip(got, ref)), per_sm
    km.close()
    Yo, sto, stao, To, floor = reference(m, T, p, Y, w["dt"], 1e-6, 1e-10,
                                         oracle.RKCK if w["method"] == kin.RKCK else oracle.RKC_POWER, energy=True)
    compare(np.vstack([ref[0], ref[1]]), np.vstack([Yo, To]), ref[2], sto, ref[3], stao, 1e-10, 1e-6, max_div_frac=0.05,
            floor=floor)


@pytest.mark.parametrize("method", [kin.RKC, kin.RKCK])
@pytest.mark.parametrize("nS,nR", [(1, 0), (7, 20), (15, 31), (16, 33), (31, 97), (32, 64), (63, 200), (64, 130), (129, 260)])
def test_energy_sizes(nS, nR, method):
    m = Mech(nS, nR, 20 * nS + nR)
    rng = np.random.default_rng(nS)
    m.cp, m.Hf = rng.uniform(20.0, 80.0, nS), rng.uniform(-1e5, 1e5, nS)
    n = 21
    T, p = rng.uniform(900.0, 1800.0, n), 101325.0 * rng.uniform(0.5, 20.0, n)
    Y = rng.uniform(0.0, 1.0, (nS, n))
    Y[0] *= 1e-9 if nS > 1 else 1.0
    if nS > 2:
        Y[2, 5] = -0.05 * Y[:, 5].sum()  # the plain FP64 path
    Y /= Y.sum(axis=0)
    T[11], T[13] = -5.0, np.nan          # not a temperature
    Yo, so, xo, _, To = oracle.integrate(oracle.Mech(m), T, p, Y, 1e-9, 1e-6, 1e-10,
                                         oracle.RKCK if method == kin.RKCK else oracle.RKC_POWER, energy=True)
    km = kin.Mechanism(m)
    Yg, Tg, sg, xg = run(km, T, p, Y, 1e-9, method, sigma=kin.SIGMA_POWER, layout=kin.LAYOUT_WARP, energy=1)
    km.close()
    assert np.array_equal(sg, so)
    ok = (so == 0) & (T > 0)
    same = ok & (xg == xo).all(axis=1)
    if nR > 1:
        assert same.sum() >= 0.9 * ok.sum()
    else:
        same = ok
    err = np.maximum((np.abs(Yg - Yo) / np.maximum(np.abs(Yo), 1e-10)).max(axis=0), np.abs(Tg - To) / np.abs(To))
    assert err[same].max() <= 1e-8, err[same].max()

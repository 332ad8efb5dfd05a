"""The lane layout's integer FP64 f (csrc/lane_int.cuh) where its records and
its grid change: one species and none of the reactions, empty reactant slots,
coefficients of 2, third bodies and falloffs, shared words that leave too
few lanes (15 / 60: the tables' f again), states on the plain FP64 path. Against the FP64 oracle over a
few steps: 1e-8 in the contract's metric on cells with the oracle's decisions,
nine cells in ten (with at most one reaction the products' number is rounding
noise, and every cell's result is compared). A call of more cells than lanes,
with as many blocks as its shared words leave room for (fewer than the grid's
with the smaller register budget), gives the same bits."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

import oracle  # noqa: E402
from paper_1309_2710_gb300 import kin  # noqa: E402
from tests.test_gpu_int_f import Mech, dev  # noqa: E402


def run(km, T, p, Y, method, **kw):
    n = T.size
    Yd = dev(Y)
    st = torch.zeros(n, dtype=torch.uint8, device="cuda")
    sta = torch.zeros((n, kin.NSTATS), dtype=torch.int32, device="cuda")
    kin.integrate(km, dev(T), dev(p), Yd, 1e-8, 1e-6, 1e-10, method, status=st, stats=sta, sigma=kin.SIGMA_POWER,
                  **kw)
    torch.cuda.synchronize()
    return Yd.cpu().numpy(), st.cpu().numpy(), sta.cpu().numpy()


@pytest.mark.parametrize("method", [kin.RKC, kin.RKCK])
@pytest.mark.parametrize("nS,nR", [(1, 0), (2, 1), (3, 30), (9, 38), (13, 12), (15, 3), (15, 60)])
def test_against_oracle(nS, nR, method):
    m = Mech(nS, nR, 7 * nS + nR)
    rng = np.random.default_rng(nS)
    n = 21
    T, p = rng.uniform(900.0, 1800.0, n), 101325.0 * rng.uniform(0.5, 20.0, n)
    Y = rng.uniform(0.0, 1.0, (nS, n))
    Y[0] *= 1e-9
    if nS > 2:
        Y[1, 3] = 0.0
        Y[2, 5] = -0.05 * Y[:, 5].sum()   # the plain FP64 path
        Y[2, 7] = -1e-7 * Y[:, 7].sum()   # a small overshoot, within the integer form
    Y /= Y.sum(axis=0)
    om = oracle.Mech(m)
    Yo, so, xo, _ = oracle.integrate(om, T, p, Y, 1e-8, 1e-6, 1e-10,
                                     oracle.RKCK if method == kin.RKCK else oracle.RKC_POWER)
    km = kin.Mechanism(m)
    # at least 64 cells per SM and a named shape: the lane layout
    served = 26 * (nS + 1) + 10 * len(m.eff) <= 448   # else the generated f above its number of cells
    few, many = 600, 6000 if served else 1200
    assert few * n >= kin.WARP_MAX_CELLS_PER_SM * torch.cuda.get_device_properties(0).multi_processor_count
    tiled = lambda k, **kw: run(km, np.tile(T, k), np.tile(p, k), np.tile(Y, (1, k)), method, **kw)
    got = tiled(few, block_threads=128, blocks_per_sm=4)
    small = tiled(few, block_threads=32, blocks_per_sm=16)
    high = [tiled(k, occupancy=kin.OCC_HIGH) for k in (few, many)]
    km.close()
    # other shapes, more cells than lanes: the same bits
    assert all(np.array_equal(x, y) for x, y in zip(got, small))
    for r, k in ((got, few), (high[0], few), (high[1], many)):
        assert np.array_equal(r[0], np.tile(r[0][:, :n], (1, k))) and np.array_equal(r[2], np.tile(r[2][:n], (k, 1)))
        assert np.array_equal(r[1], np.tile(so, k))
    assert np.array_equal(high[0][0][:, :n], high[1][0][:, :n]) and np.array_equal(high[0][2][:n], high[1][2][:n])
    Yg, xg = got[0][:, :n], got[2][:n]
    same = (xg == xo).all(axis=1)
    if nR > 1:
        assert same.mean() >= 0.9, same.mean()
    else:
        same[:] = True
    err = np.abs(Yg - Yo) / np.maximum(np.abs(Yo), 1e-10)
    assert err[:, same].max() <= 1e-8, err[:, same].max()

"""The warp layout's integer FP64 f (csrc/warp_int.cuh) at the sizes where its
tables and groups change: species around 16, 32, 64 and 128, reactions around
multiples of the lanes and of the chunks, empty reactant slots, coefficients
of 2, efficiencies of 0 and far apart, and states that take the plain FP64 path
(a concentration below -2^-9 of the total). Against the FP64 oracle over a few
steps: 1e-8 in the contract's metric on cells with the oracle's decisions,
nine cells in ten. With at most one reaction the spectral radius is rounding
noise (f is linear along every direction the power method sees), and with it
the number of products: there every cell's result is compared instead."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

import oracle  # noqa: E402
from paper_1309_2710_gb300 import kin  # noqa: E402


class Mech:
    """Random reactions over random species (mass is not conserved: W is free)."""

    def __init__(self, nS, nR, seed):
        rng = np.random.default_rng(seed)
        self.W = rng.uniform(2.0, 60.0, nS)
        self.reac = rng.integers(-1 if nS > 3 else 0, nS, (nR, 2)).astype(np.int32)
        self.prod = rng.integers(-1, nS, (nR, 2)).astype(np.int32)
        two = rng.uniform(size=nR) < 0.2
        self.reac[two, 1] = self.reac[two, 0]
        order = (self.reac >= 0).sum(1)
        # rates of a few 1e5 / s per mass fraction at C ~ 1e-5 mol / cm^3
        self.lnA = np.log(10.0) * rng.uniform(2.0, 5.0, nR) + 5.0 * np.log(10.0) * (order - 1)
        self.beta, self.Ea = rng.uniform(-0.2, 0.2, nR), rng.uniform(0.0, 1e4, nR)
        self.rtype = rng.choice([0, 0, 0, 1, 2], nR).astype(np.int8)
        self.lnA[self.rtype == 1] += 5.0 * np.log(10.0)
        rows = int((self.rtype > 0).sum())
        self.eff = rng.uniform(0.5, 3.0, (rows, nS))
        self.eff[rng.uniform(size=(rows, nS)) < 0.2] = 0.0
        if rows > 1:
            self.eff[0] = 0.0           # only a trace species collides
            self.eff[0, 0] = 1.0
            self.eff[1, ::2] *= 1e-9
        self.lnA0, self.beta0, self.Ea0 = self.lnA + 11.0, self.beta.copy(), 0.8 * self.Ea
        plain = self.rtype != 2
        self.lnA0[plain] = self.beta0[plain] = self.Ea0[plain] = 0.0
        self.n_species, self.n_reactions = nS, nR


def dev(a):
    return torch.as_tensor(np.ascontiguousarray(a), device="cuda")


@pytest.mark.parametrize("method", [kin.RKC, kin.RKCK])
@pytest.mark.parametrize("nS,nR", [(1, 0), (2, 1), (15, 31), (16, 33), (17, 64), (32, 255), (33, 257), (64, 512),
                                   (65, 513), (111, 1030), (129, 300), (200, 1100)])
def test_sizes_against_oracle(nS, nR, method):
    m = Mech(nS, nR, 10 * nS + nR)
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
    meth = oracle.RKCK if method == kin.RKCK else oracle.RKC_POWER
    dt = 1e-8
    Yo, so, xo, _ = oracle.integrate(om, T, p, Y, dt, 1e-6, 1e-10, meth)
    km = kin.Mechanism(m)
    got = []
    for threads in (128, 32):
        Yd = dev(Y)
        st = torch.zeros(n, dtype=torch.uint8, device="cuda")
        sta = torch.zeros((n, kin.NSTATS), dtype=torch.int32, device="cuda")
        kin.integrate(km, dev(T), dev(p), Yd, dt, 1e-6, 1e-10, method, status=st, stats=sta,
                      sigma=kin.SIGMA_POWER, layout=kin.LAYOUT_WARP, block_threads=threads)
        torch.cuda.synchronize()
        got.append((Yd.cpu().numpy(), st.cpu().numpy(), sta.cpu().numpy()))
    km.close()
    # one warp or several per cell: the same bits
    assert all(np.array_equal(a, b) for a, b in zip(*got))
    Yg, sg, xg = got[0]
    assert np.array_equal(sg, so)
    same = (xg == xo).all(axis=1)
    err = np.abs(Yg - Yo) / np.maximum(np.abs(Yo), 1e-10)
    if nR > 1:
        assert same.mean() >= 0.9, same.mean()
    else:
        same[:] = True
    assert err[:, same].max() <= 1e-8, err[:, same].max()


@pytest.mark.parametrize("nS,nR", [(2, 1), (9, 38), (15, 31), (16, 33)])
def test_lanes_per_cell_do_not_change_the_bits(nS, nR):
    """A call of many cells gives each a quarter warp, one of few half a warp."""
    m = Mech(nS, nR, 5 * nS + nR)
    rng = np.random.default_rng(nS)
    n, tiles = 37, 400
    T, p = rng.uniform(900.0, 1800.0, n), 101325.0 * rng.uniform(0.5, 20.0, n)
    Y = rng.uniform(0.0, 1.0, (nS, n))
    if nS > 2:
        Y[2, 5] = -0.05 * Y[:, 5].sum()
    Y /= Y.sum(axis=0)
    assert n * tiles > kin.WARP_MAX_CELLS_PER_SM * torch.cuda.get_device_properties(0).multi_processor_count
    km = kin.Mechanism(m)
    for sigma in (kin.SIGMA_POWER, kin.SIGMA_GERSHGORIN):
        got = []
        for k in (1, tiles):
            Yd = dev(np.tile(Y, (1, k)))
            st = torch.zeros(n * k, dtype=torch.uint8, device="cuda")
            sta = torch.zeros((n * k, kin.NSTATS), dtype=torch.int32, device="cuda")
            kin.integrate(km, dev(np.tile(T, k)), dev(np.tile(p, k)), Yd, 1e-7, 1e-6, 1e-10, kin.RKC, status=st,
                          stats=sta, sigma=sigma)
            torch.cuda.synchronize()
            got.append((Yd.cpu().numpy(), st.cpu().numpy(), sta.cpu().numpy()))
        one, many = got
        assert np.array_equal(np.tile(one[0], (1, tiles)), many[0])
        assert np.array_equal(np.tile(one[1], tiles), many[1]) and np.array_equal(np.tile(one[2], (tiles, 1)), many[2])
    km.close()

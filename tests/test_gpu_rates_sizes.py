"""kin.rates in FP64 at the sizes where its lanes per cell change (8, 16 and 32
species, 24 and 40 reactions), species by species against extended precision:
the bounds of test_int_f_species.py, and a rounding per species for third-body
sums that are taken in FP64 (only a trace species collides)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

from paper_1309_2710_gb300 import kin, synth  # noqa: E402
from tests import int_f_replay  # noqa: E402
from tests.test_gpu_int_f import Mech, dev  # noqa: E402
from tests.test_int_f_species import ULP  # noqa: E402


@pytest.mark.parametrize("nS,nR", [(1, 0), (2, 1), (7, 23), (8, 24), (9, 23), (16, 23), (16, 24), (17, 39), (17, 40),
                                   (31, 39), (32, 1), (33, 39), (65, 100), (129, 300)])
def test_sizes(nS, nR):
    m = Mech(nS, nR, 3 * nS + nR)
    f = int_f_replay.Mech(None, m)
    rng = np.random.default_rng(nS)
    n = 37
    T, p = rng.uniform(500.0, 2500.0, n), 101325.0 * rng.uniform(0.5, 20.0, n)
    Y = rng.uniform(0.0, 1.0, (nS, n)) * 10.0 ** rng.uniform(-9, 0, (nS, n))
    if nS > 2:
        Y[1, 3] = 0.0
        Y[2, 7] = -1e-7 * Y[:, 7].sum()
    Y /= Y.sum(axis=0)
    km = kin.Mechanism(m)
    out = kin.rates(km, dev(T), dev(p), dev(Y), kin.FP64).cpu().numpy()
    many = kin.rates(km, dev(np.tile(T, 900)), dev(np.tile(p, 900)), dev(np.tile(Y, (1, 900))), kin.FP64).cpu().numpy()
    km.close()
    assert np.array_equal(many, np.tile(out, (1, 900)))
    for c in range(n):
        ref, mag = f.reference(T[c], p[c], Y[:, c])
        big = (abs(m.lnA) + abs(m.beta) * np.log(T[c]) + m.Ea / (synth.R_GAS * T[c])).max(initial=0.0)
        assert (np.abs(out[:, c] - ref) <= ULP * (16 + nS + 4 * big) * mag).all(), c

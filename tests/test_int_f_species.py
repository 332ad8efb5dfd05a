"""The integer FP64 f species by species: on unburnt mixtures, whose radicals are
far below the major species, every species' rate against extended precision
and relative to the sum of its own |nu_ij Omega_j|, not to the cell's largest
rate. Bounds: with given rate constants 16 roundings of 2^-53 (products, third-body
sum, sum of a row, molar masses); the rate constants from T add their exponent's,
four roundings of the sum of its |terms|."""
import numpy as np
import pytest

from paper_1309_2710_gb300 import synth
from tests import int_f_replay

ULP = 2.0 ** -53
# radicals log-uniform between these powers of ten; None: exactly zero
RADICALS = [(-16, -6), (-20, -8), (-30, -10), (-60, -30), None]


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    L = int_f_replay.build(tmp_path_factory.mktemp("replay"))
    if L is None:
        pytest.skip("g++ not available")
    return L


def unburnt(wl, m, n, radicals):
    """Three major species of the workload's mixture, the rest as radicals; one
    cell in four with a small negative one."""
    rng = np.random.default_rng(11)
    _, _, Y = synth.workload_states(wl, m, cells=n)
    for c in range(n):
        major = np.argsort(Y[:, c])[-3:]
        y = Y[major, c]
        Y[:, c] = 0.0 if radicals is None else 10.0 ** rng.uniform(*radicals, m.n_species)
        if c % 4 == 3:
            Y[rng.integers(m.n_species), c] *= -1.0
        Y[major, c] = y
    return rng.uniform(700.0, 1500.0, n), 101325.0 * rng.uniform(1.0, 20.0, n), Y / Y.sum(axis=0)


@pytest.mark.parametrize("radicals", RADICALS)
@pytest.mark.parametrize("wl", ["h2_9sp_rkck", "h2co_13sp_rkc", "ch4_53sp_rkc_mixed", "c2h4_111sp_rkc_batched"])
def test_unburnt(lib, wl, radicals):
    m = synth.workload_mechanism(wl)
    f = int_f_replay.Mech(lib, m)
    n = 8 if m.n_species > 50 else 24
    T, p, Y = unburnt(wl, m, n, radicals)
    for c in range(n):
        cell = T[c], p[c], Y[:, c]
        bound = ULP * (16 + 4 * (abs(m.lnA) + abs(m.beta) * np.log(T[c]) + m.Ea / (synth.R_GAS * T[c])).max())
        ref, mag = f.reference(*cell)
        out, scale = f.warp(*cell, -(c % 2))  # (-1: the scale is estimated first)
        assert (np.abs(out - ref) <= bound * mag).all(), (c, float((np.abs(out - ref) / np.maximum(mag, 1e-300)).max()))
        if m.n_species > 16:
            continue
        ref, mag = f.reference(*cell, k=f.constants(T[c]))
        out, plain = f.lane(*cell)
        assert plain == 0
        assert (np.abs(out - ref) <= 16 * ULP * mag).all(), (c, float((np.abs(out - ref) / np.maximum(mag, 1e-300)).max()))

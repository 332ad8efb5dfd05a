"""The integer FP64 f species by species: on unburnt mixtures, whose radicals are
far below the major species, every species' rate against extended precision
and relative to the sum of its own |nu_ij Omega_j|, not to the cell's largest
rate. Bounds: with given rate constants 16 roundings of 2^-53 (products, third-body
sum, sum of a row, molar masses); the rate constants from T add their exponent's,
four roundings of the sum of its |terms|. Third-body sums with efficiencies far
apart are held to the error of the plain FP64 form."""
import types

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


def third_bodies(nS, top, rtype, rng):
    """A -> B with a third body or a falloff for every species, k = 1, efficiencies
    of 0.7 to 3 and `top` for the first species."""
    n = nS
    z = np.zeros(n)
    m = types.SimpleNamespace(n_species=nS, n_reactions=n, W=rng.uniform(2.0, 60.0, n), lnA=z, beta=z, Ea=z,
                              reac=np.full((n, 2), -1), prod=np.full((n, 2), -1), rtype=np.full(n, rtype),
                              lnA0=z + 10.0, beta0=z, Ea0=z, eff=rng.uniform(0.5, 3.0, (n, nS)))
    m.prod[:, 0], m.reac[:, 0] = np.arange(n), (np.arange(n) + 1) % n
    m.eff[:, 0], m.eff[:, 1] = top, 0.7
    return m


def plain(f, T, p, Y):
    """The same rates in FP64: two interleaved partial sums per third body."""
    m = f.m
    k, k0 = f.constants(T)
    s, Ctot = (Y * (1.0 / m.W)).sum(), p * 1e-6 / (synth.R_GAS * T)
    C = Y * (1.0 / m.W) * (Ctot * (1.0 / s))
    part = np.zeros((2, m.n_reactions))
    for i in range(m.n_species):
        part[i % 2] += m.eff[:, i] * C[i]
    M = part[0] + part[1]
    if m.rtype[0] == 2:
        M = k0 * M
        M /= 1.0 + M
    q = k * C[m.reac[:, 0]] * M
    out = np.zeros(m.n_species)
    out[m.prod[:, 0]] += q
    out[m.reac[:, 0]] -= q
    return out * m.W * (s * (1.0 / Ctot))


@pytest.mark.parametrize("rtype", [1, 2])
@pytest.mark.parametrize("top", [3.0, 12.0, 50.0, 200.0])
@pytest.mark.parametrize("nS,n", [(13, 200), (111, 30)])
def test_third_body_error(lib, nS, n, top, rtype):
    rng = np.random.default_rng(9)
    f = int_f_replay.Mech(lib, third_bodies(nS, top, rtype, rng))
    err = {"warp": [], "lane": [], "plain": []}
    for c in range(n):
        Y = rng.uniform(0.0, 1.0, nS) * 10.0 ** rng.uniform(-6, 0, nS)
        Y[0] = 1e-7
        cell = rng.uniform(800.0, 1200.0), 101325.0 * rng.uniform(0.5, 2.0), Y / Y.sum()
        ref, mag = f.reference(*cell)
        err["warp"].append((f.warp(*cell, 0)[0] - ref) / mag)
        err["plain"].append((plain(f, *cell) - ref) / mag)
        if nS <= 16:
            out, general = f.lane(*cell)
            if not general:  # (top = 200: the whole cell in plain FP64)
                err["lane"].append((out - ref) / mag)
    rms = {k: float(np.sqrt(np.mean(np.square(v)))) for k, v in err.items() if v}
    # two rms values of some 3,000 samples each: 5 % between them by chance (3 sigma)
    for k, v in rms.items():
        assert v <= 1.1 * rms["plain"], {k: v / ULP for k, v in rms.items()}


@pytest.mark.parametrize("wl", ["h2_9sp_rkck", "h2co_13sp_rkc", "ch4_53sp_rkc_mixed"])
def test_plain_path(lib, wl):
    """States outside the integer forms' range (a species at -0.05 to -300 of the
    total, as in a step that blew up): plain FP64, whose sums of up to 64 terms and
    species add their roundings to the bound."""
    m = synth.workload_mechanism(wl)
    f = int_f_replay.Mech(lib, m)
    T, p, Y = unburnt(wl, m, 8, (-6, -2))
    for c in range(8):
        Y[c % m.n_species, c] = -10.0 ** (c / 2.0 - 1.3) * Y[:, c].sum()
        if c % 2:
            Y[(c + 3) % m.n_species, c] = 1.5 * abs(Y[:, c]).sum()
        cell = T[c], p[c], Y[:, c] / Y[:, c].sum()
        bound = ULP * (16 + 64 + m.n_species + 4 * (abs(m.lnA) + abs(m.beta) * np.log(T[c]) + m.Ea / (synth.R_GAS * T[c])).max())
        ref, _ = f.reference(*cell)
        _, mag = f.reference(cell[0], cell[1], abs(cell[2]))
        # (the terms' size at these concentrations; the mixture sum cancels)
        w = abs(cell[2] / m.W).sum() / abs((cell[2] / m.W).sum())
        out, _ = f.warp(*cell, 0)
        assert (np.abs(out - ref) <= bound * w ** 4 * mag).all(), c

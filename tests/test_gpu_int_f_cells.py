"""A cell's bits do not depend on the cells around it: kin.rates and the energy
equation in the warp layout (RKC and RKCK), on cells whose largest rates lie
many octaves apart, alone, permuted and among others, and with fewer groups of
lanes than cells, so that each serves several."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

from paper_1309_2710_gb300 import kin, synth  # noqa: E402


def dev(a):
    return torch.as_tensor(np.ascontiguousarray(a), device="cuda")


def cells(wl, m, n):
    rng = np.random.default_rng(3)
    _, _, Y = synth.workload_states(wl, m, cells=n)
    for c in range(n):
        major = np.argsort(Y[:, c])[-3:]
        y = Y[major, c]
        Y[:, c] = 10.0 ** rng.uniform(-12, -3, m.n_species)
        Y[major, c] = y
    return rng.uniform(500.0, 2500.0, n), 101325.0 * 10.0 ** rng.uniform(-1, 1.3, n), Y / Y.sum(axis=0)


@pytest.mark.parametrize("wl", ["h2_9sp_rkck", "h2co_13sp_rkc", "ch4_53sp_rkc_mixed", "c2h4_111sp_rkc_batched"])
def test_rates(wl):
    m = synth.workload_mechanism(wl)
    n = 20011 if m.n_species < 50 else 3011
    T, p, Y = cells(wl, m, n)
    km = kin.Mechanism(m)
    f = lambda at: kin.rates(km, dev(T[at]), dev(p[at]), dev(Y[:, at]), kin.FP64).cpu().numpy()
    every = f(np.arange(n))
    at = np.random.default_rng(1).permutation(n)
    assert np.array_equal(f(at), every[:, at])
    few = at[:5]
    assert np.array_equal(f(few), every[:, few])
    km.close()


@pytest.mark.parametrize("wl,method,dt", [("h2co_13sp_rkc", kin.RKC, 1e-8), ("h2_9sp_rkck", kin.RKCK, 1e-9),
                                          ("ch4_53sp_rkc_mixed", kin.RKC, 1e-9)])
def test_energy(wl, method, dt):
    m = synth.workload_mechanism(wl + "_energy")
    n = 12011 if m.n_species < 50 else 1511
    T, p, Y = cells(wl, m, n)
    km = kin.Mechanism(m)

    def run(at, **kw):
        Td, Yd = dev(T[at]), dev(Y[:, at])
        st = torch.zeros(len(at), dtype=torch.uint8, device="cuda")
        sta = torch.zeros((len(at), kin.NSTATS), dtype=torch.int32, device="cuda")
        kin.integrate(km, Td, dev(p[at]), Yd, dt, 1e-6, 1e-10, method, status=st, stats=sta, sigma=kin.SIGMA_POWER,
                      energy=1, layout=kin.LAYOUT_WARP, **kw)
        return [a.cpu().numpy() for a in (Td, Yd.T, st, sta)]

    every = run(np.arange(n))
    at = np.random.default_rng(1).permutation(n)
    for got, i in ((run(at), at), (run(at[:5]), at[:5]), (run(np.arange(n), block_threads=32, blocks_per_sm=1), np.arange(n))):
        for a, b in zip(got, every):
            assert np.array_equal(a, b[i], equal_nan=a.dtype.kind == "f")
    km.close()

"""The warp layout's limit on a mechanism does not depend on the lanes that a call
gives each cell: 16 species with 2,000 reactions are taken at any number of
cells (a whole, half and a quarter warp per cell), with the same bits."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

from paper_1309_2710_gb300 import kin  # noqa: E402
from tests.test_gpu_int_f import Mech, dev  # noqa: E402


@pytest.mark.parametrize("threads", [0, 256])
def test_many_reactions(threads):
    m = Mech(16, 2000, 4)
    rng = np.random.default_rng(2)
    n = 19
    T, p = rng.uniform(900.0, 1800.0, n), 101325.0 * rng.uniform(0.5, 20.0, n)
    Y = rng.uniform(0.0, 1.0, (16, n))
    Y /= Y.sum(axis=0)
    sm = torch.cuda.get_device_properties(0).multi_processor_count
    km = kin.Mechanism(m)
    got = []
    for k in (1, sm, 4 * sm):  # 19 cells, 19 and 76 per SM
        Yd = dev(np.tile(Y, (1, k)))
        sta = torch.zeros((n * k, kin.NSTATS), dtype=torch.int32, device="cuda")
        kin.integrate(km, dev(np.tile(T, k)), dev(np.tile(p, k)), Yd, 1e-10, 1e-6, 1e-10, kin.RKC, stats=sta,
                      sigma=kin.SIGMA_POWER, layout=kin.LAYOUT_WARP, block_threads=threads)
        Yg, x = Yd.cpu().numpy(), sta.cpu().numpy()
        assert np.array_equal(Yg, np.tile(Yg[:, :n], (1, k))) and np.array_equal(x, np.tile(x[:n], (k, 1)))
        got.append((Yg[:, :n], x[:n]))
    km.close()
    assert all(np.array_equal(a, b) for g in got[1:] for a, b in zip(g, got[0]))

"""Mixed-precision RKC of a small mechanism in the warp layout, whose rate
constants are staged in shared memory: with an odd number of 8-byte words of
them, the words of every second cell of a block must still begin on the 16
bytes that the FP32 efficiency sums load at once. Against the lane layout's
mixed path, whose arithmetic is the same to FP32 rounding: 1e-5 in the
contract's metric, as between either and the oracle."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

from paper_1309_2710_gb300 import kin, synth  # noqa: E402
from tests.test_gpu_int_f import dev  # noqa: E402


@pytest.mark.parametrize("nR", [53, 54, 55, 56])
def test_odd_staged_words(nR):
    m = synth.make_mechanism(13, nR, ("C", "H", "O", "N"), tb_frac=0.2, fo_frac=0.1, seed=31)
    n = 301
    T, p, Y = synth.make_states(m, n, T_range=(1100.0, 1500.0), seed=32)
    km = kin.Mechanism(m)
    out = []
    for layout in (kin.LAYOUT_LANE, kin.LAYOUT_WARP):
        Yd = dev(Y)
        st = torch.zeros(n, dtype=torch.uint8, device="cuda")
        kin.integrate(km, dev(T), dev(p), Yd, 1e-8, 1e-6, 1e-10, kin.RKC, kin.MIXED, status=st,
                      sigma=kin.SIGMA_POWER, layout=layout)
        torch.cuda.synchronize()
        assert not st.any().item()
        out.append(Yd.cpu().numpy())
    km.close()
    a, b = out
    assert (np.abs(a - b) / np.maximum(np.abs(a), 1e-10 / 1e-6)).max() <= 1e-5

"""The FP32 D3Q27 step that loads f' one plane ahead (items of 5 planes and
more) and the one that does not hold bitwise the state of the reference pair."""
import numpy as np
import pytest

from paper_2101_06769_gb300 import Domain
from paper_2101_06769_gb300.lbmp import OPT_CHUNK, OPT_KERNEL

pytestmark = pytest.mark.gpu

PHYS = dict(rho_ratio=3.0, nu_ratio=1.0, nu_h=0.05, g_accel=1e-5, L_ref=32.0, mobility=0.02, width=4.0)


# items on both sides of the switch, one item per column, a last item of one
# plane, and the automatic choice where it loads ahead in several rounds
@pytest.mark.parametrize("dims,periodic,chunk", [
    ((37, 11, 13), (1, 1, 0), 4), ((37, 11, 13), (1, 1, 0), 5), ((37, 11, 13), (1, 1, 1), 6), ((37, 11, 13), (1, 1, 0), 13),
    ((32, 4, 11), (1, 1, 1), 5), ((5, 3, 64), (1, 1, 0), 0), ((72, 72, 72), (1, 1, 0), 0), ((130, 66, 131), (1, 1, 1), 0)])
def test_loading_ahead_is_bitwise_the_reference_pair(dims, periodic, chunk):
    out = []
    for kernel in (0, 1):
        d = Domain(3, dims, periodic, **PHYS)
        d.set_option(OPT_KERNEL, kernel)
        if kernel == 0:
            d.set_option(OPT_CHUNK, chunk)
        d.init("rt", [dims[2] / 2, 1.5, 1e-2, 1.0], seed=4)
        d.step(3)
        out.append(d.get_state())
        d.close()
    for a, b in zip(*out):
        assert np.isfinite(a).all() and np.array_equal(a, b)

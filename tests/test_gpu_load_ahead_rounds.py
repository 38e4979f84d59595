"""The FP32 D3Q27 step that loads f' one plane ahead, where the grid takes
several rounds of work items (a CTA goes from one item to the next), holds
bitwise the state of the reference pair.  test_launch_rules_cpu.py asserts that
these domains are stepped so."""
import numpy as np
import pytest

from paper_2101_06769_gb300 import Domain
from paper_2101_06769_gb300.lbmp import OPT_KERNEL

pytestmark = pytest.mark.gpu

PHYS = dict(rho_ratio=3.0, nu_ratio=1.0, nu_h=0.05, g_accel=1e-5, L_ref=32.0, mobility=0.02, width=4.0)

# ragged in x and y, a last item shorter than the others
DOMAINS = [((121, 126, 115), (1, 1, 0)), ((127, 122, 128), (1, 1, 1))]


@pytest.mark.parametrize("dims,periodic", DOMAINS)
def test_several_rounds_are_bitwise_the_reference_pair(dims, periodic):
    out = []
    for kernel in (0, 1):
        d = Domain(3, dims, periodic, **PHYS)
        d.set_option(OPT_KERNEL, kernel)
        d.init("rt", [dims[2] / 2, 1.5, 1e-2, 1.0], seed=4)
        d.step(3)
        out.append(d.get_state())
        d.close()
    for a, b in zip(*out):
        assert np.isfinite(a).all() and np.array_equal(a, b)

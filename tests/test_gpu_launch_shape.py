"""The default planes (rows) per work item change speed only: a domain stepped
with them holds bitwise the state of the same domain stepped with the whole
marching axis as one work item."""
import numpy as np
import pytest

from paper_2101_06769_gb300 import Domain
from paper_2101_06769_gb300.lbmp import OPT_CHUNK

pytestmark = pytest.mark.gpu

PHYS = dict(rho_ratio=3.0, nu_ratio=1.0, nu_h=0.05, g_accel=1e-5, L_ref=32.0, mobility=0.02, width=4.0)


# one plane per item, a few planes with a remainder, a domain just below and
# just above three rounds of the full grid, and the smallest extents
@pytest.mark.parametrize("dims,flags,storage", [
    ((2, 2, 1), 0, 0), ((64, 256, 1), 0, 0), ((130, 67, 1), 8, 0), ((1350, 301, 1), 0, 2),
    ((2, 2, 2), 0, 0), ((33, 5, 7), 0, 0), ((64, 64, 29), 0, 0), ((66, 64, 29), 8, 0), ((66, 64, 29), 0, 1),
    ((128, 128, 113), 0, 0), ((128, 128, 115), 0, 0)])
def test_default_items_are_bitwise_one_item_per_column(dims, flags, storage):
    D = 2 if dims[2] == 1 else 3
    periodic = (1, 1, 0) if D == 3 else (1, 0, 1)
    out = []
    for chunk in (0, dims[D - 1]):
        d = Domain(D, dims, periodic, storage=storage, flags=flags, **PHYS)
        d.set_option(OPT_CHUNK, chunk)
        d.init("rt", [dims[D - 1] / 2, 1.5, 1e-2, 1.0], seed=4)
        d.step(3)
        out.append(d.get_state())
        d.close()
    for a, b in zip(*out):
        assert np.isfinite(a).all() and np.array_equal(a, b)

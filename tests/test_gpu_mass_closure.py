"""The collision keeps each cell's sum of g also where the populations have
mixed signs and nearly cancel (a bulk with phi near 0).

A uniform state: each half of the directions adds up to the negative of the
other, in another order, with edges and corners 1000 times the faces.  The
stored rest population is then about 1e-6, so what the stored populations add
up to is off the cell's phi only by the rounding of that value (6e-14) and of the
compensation (13 terms of at most 3e-6 in FP32, 2e-12): 1e-11."""
import math

import numpy as np
import pytest

from paper_2101_06769_gb300 import Domain
from paper_2101_06769_gb300.lbmp import FLAG_AA, OPT_KERNEL

pytestmark = pytest.mark.gpu

PHYS = dict(rho_ratio=20.0, nu_ratio=2.0, nu_h=0.05, sigma=1e-2, L_ref=8.0, mobility=0.02, width=4.0)


def mixed_signs(D, rng):
    c = [(x, y, z) for z in ((-1, 0, 1) if D == 3 else (0,)) for y in (-1, 0, 1) for x in (-1, 0, 1)]
    half = len(c) // 2
    g = np.zeros(len(c))
    for order in range(1, D + 1):  # faces, edges, corners
        dirs = [a for a in range(half) if sum(map(abs, c[a])) == order]
        v = (rng.standard_normal(len(dirs)) * (1e-3 if order == 1 else 1.0)).astype(np.float32)
        g[dirs] = v
        g[[len(c) - 1 - a for a in dirs]] = -rng.permutation(v)
    g[half] = np.float32(1e-6 - math.fsum(g))
    return g


@pytest.mark.parametrize("D,dims,flags,kernel", [(3, (33, 5, 7), 0, 0), (3, (33, 5, 7), 0, 1), (3, (33, 5, 7), FLAG_AA, 0),
                                                 (2, (33, 7, 1), 0, 0), (2, (33, 7, 1), 0, 1)])
def test_collision_keeps_the_sum_of_g(D, dims, flags, kernel):
    rng = np.random.default_rng(7)
    for _ in range(12):
        d = Domain(D, dims, (1, 1, 1), flags=flags, **PHYS)
        if kernel:
            d.set_option(OPT_KERNEL, kernel)
        f = np.zeros(d.shape)
        g = np.broadcast_to(mixed_signs(D, rng).reshape(-1, 1, 1, 1), d.gshape)
        d.set_state(f, g)
        phi = d.get_phi()
        d.step(1)
        _, g, _ = d.get_state()
        d.close()
        cells = g.reshape(g.shape[0], -1)
        assert abs(cells).max() > 1e4 * abs(cells[cells.shape[0] // 2]).max()  # nearly cancelled
        for k in (0, cells.shape[1] // 2, cells.shape[1] - 1):
            assert abs(math.fsum(cells[:, k]) - phi.ravel()[k]) <= 1e-11

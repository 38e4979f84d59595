"""The observables over the whole range of FP32 velocities, and their sums over
thousands of cells per thread: as exact as FP64 per cell.

A cell at rest density 1 whose only population is v in direction +x has
u = 3 v; u, its square and the sums are compared with the same in Python's
FP64.  Tolerances: u is formed in FP32 (two roundings, 2e-7); a sum of n terms
in FP64 is off by at most n 2^-53 of the sum of their magnitudes, and a term by
8 roundings."""
import math

import numpy as np
import pytest

import device_functions
from paper_2101_06769_gb300 import FLAG_PHASE_REDUCED, Domain
from paper_2101_06769_gb300.lbmp import FLAG_AA

pytestmark = pytest.mark.gpu

PHYS = dict(rho_ratio=20.0, nu_ratio=2.0, nu_h=0.05, sigma=1e-2, L_ref=8.0, mobility=0.02, width=4.0)


# one march (FP32 D3Q27), and the phi pass with gathers (in place, 2-D, a symmetry axis)
@pytest.mark.parametrize("D,dims,periodic,flags", [
    (3, (33, 5, 7), (1, 1, 0), 0), (3, (5, 6, 70), (1, 1, 1), FLAG_PHASE_REDUCED), (3, (33, 5, 7), (1, 1, 0), FLAG_AA),
    (2, (33, 7, 1), (1, 0, 1), 0), (2, (33, 7, 1), (2, 0, 1), 0)])
@pytest.mark.parametrize("u,health", [(math.inf, 3), (1e20, 2), (3.0, 2), (1e-3, 0), (1e-17, 0), (1e-22, 0), (1e-25, 0)])
def test_one_moving_cell(D, dims, periodic, flags, u, health):
    d = Domain(D, dims, periodic, flags=flags, **PHYS)
    d.init("uniform", [1.0, 0.0, 0.0, 0.0, 0.0])
    f, g, _ = d.get_state()
    f[:] = 0.0
    f[(14, 2, 2, 2) if D == 3 else (5, 0, 3, 2)] = 1e39 if math.isinf(u) else u / 3.0
    d.set_state(f, g)
    ob = d.observables()
    d.close()
    assert ob.health == health
    if math.isinf(u):
        assert ob.max_u == math.inf and ob.kinetic_energy == math.inf
    else:
        assert abs(ob.max_u / u - 1.0) < 1e-6
        assert abs(ob.kinetic_energy / (0.5 * u * u) - 1.0) < 1e-6


@pytest.fixture(scope="module")
def functions(tmp_path_factory):
    return device_functions.load(tmp_path_factory.mktemp("device_functions"))


@pytest.mark.parametrize("n", [1, 26, 2048, 6000])
def test_sums_of_many_cells_per_thread(functions, n):
    rng = np.random.default_rng(n)
    hi = rng.uniform(0.1, 1.0, n).astype(np.float32)
    phi = np.stack([hi, (hi * rng.uniform(-2.0**-25, 2.0**-25, n)).astype(np.float32)], 1)
    rho = rng.uniform(0.05, 1.0, n).astype(np.float32)
    u = (1e-3 * rng.standard_normal((n, 3))).astype(np.float32)
    ph = rng.standard_normal(n).astype(np.float32)
    out = np.empty(4)
    assert functions.obs_sums(n, *(a.ctypes.data_as(device_functions.ctypes.c_void_p) for a in (phi, rho, u, ph, out))) == 0
    uu = (u.astype(float) ** 2).sum(1)
    eps = 2.0**-53
    mass = 128 * math.fsum(phi.astype(float).ravel())  # 128 threads take the same cells
    energy = 128 * 0.5 * math.fsum(rho.astype(float) * uu)
    assert abs(out[0] / mass - 1.0) <= (n + 16) * eps
    assert abs(out[1] / energy - 1.0) <= (n + 16) * eps
    assert abs(out[2] / math.sqrt(uu.max()) - 1.0) <= 8 * eps
    assert out[3] == 0.0

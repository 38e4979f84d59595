"""The observables taken in one march over an FP32 D3Q27 domain against the phi
pass and gathers, which the in-place storage form (the same populations after
lbmp_init) still runs, and against sums over the exchange state.

Tolerances: both paths form every per-cell value by the same FP32 operations,
compiled apart (a few ulps of the terms, 1e-6 of the result), and sum to FP64
accuracy (mass: 1e-12 of the total)."""
import numpy as np
import pytest

from paper_2101_06769_gb300 import FLAG_PHASE_REDUCED, Domain
from paper_2101_06769_gb300.lbmp import FLAG_AA

pytestmark = pytest.mark.gpu

PHYS = dict(rho_ratio=20.0, nu_ratio=2.0, nu_h=0.05, sigma=1e-2, U0=0.01, L_ref=8.0, mobility=0.02, width=4.0)

# thinnest extents, a single ragged tile, tile edges, several work items per CTA
DIMS = [(2, 2, 2), (3, 2, 5), (31, 3, 2), (33, 5, 17), (32, 4, 9), (65, 29, 23), (160, 96, 130)]


@pytest.mark.parametrize("walls", [0, 1])
@pytest.mark.parametrize("dims", DIMS)
def test_march_matches_gathers(dims, walls):
    obs = []
    for flags in (0, FLAG_AA):
        d = Domain(3, dims, (1, 1, 1 - walls), flags=flags, **PHYS)
        if walls:
            d.init("rt", [dims[2] / 2, 1.0, 1e-2, 0.0], seed=3)
        else:
            d.init("drop_static", [0.3 * min(dims), 1.0, 1e-2], seed=3)
        obs.append(d.observables().as_dict())
        d.close()
    a, b = obs
    assert a["health"] == b["health"] == 0 and a["step"] == b["step"] == 0
    assert a["mass_drift_rel"] == 0.0
    assert abs(a["mass"] / b["mass"] - 1) < 1e-12
    p_scale = max(abs(b["p_in"]), abs(b["p_out"]), 1e-12)
    for k in ("p_in", "p_out", "laplace_dp"):
        assert abs(a[k] - b[k]) <= 1e-6 * p_scale, k
    for k in ("kinetic_energy", "max_u"):
        assert abs(a[k] - b[k]) <= 1e-6 * abs(b[k]), k
    for k in ("tip_spike", "tip_bubble"):
        assert abs(a[k] - b[k]) <= 1e-9, k


@pytest.mark.parametrize("dims", [(3, 2, 5), (33, 5, 17), (130, 64, 70)])
@pytest.mark.parametrize("flags", [0, FLAG_PHASE_REDUCED])
def test_march_after_steps_matches_the_exchange_state(dims, flags):
    d = Domain(3, dims, (1, 1, 0), flags=flags, **PHYS)
    d.init("rt", [dims[2] / 2, 1.0, 1e-2, 0.0], seed=5)
    for n in (1, 2):
        d.step(n)
        _, g, _ = d.get_state()
        ob = d.observables()
        assert ob.health == 0
        assert abs(ob.mass / g.sum() - 1) < 1e-12
        assert abs(ob.mass_drift_rel) < 1e-7
    d.close()


def test_march_counts_non_finite_cells():
    d = Domain(3, (33, 9, 12), (1, 1, 1), **PHYS)
    d.init("drop_static", [3.0, 0.0, 1e-2], seed=1)
    f, g, _ = d.get_state()
    for bad in (np.nan, np.inf):
        h = f.copy()
        h[4, 5, 6, 32] = bad
        d.set_state(h, g)
        assert d.observables().health & 1
    d.set_state(f, g)
    assert d.observables().health == 0
    d.close()

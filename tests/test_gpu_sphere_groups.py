"""The adjoint's sphere groups (8, 16 or 32 spheres per warp step; every second
sphere per lane of a pair) against the oracle at their edges: a sphere that is
left out or counted twice would move its own sums by all of their value."""

import numpy as np
import pytest

from oracle import shs_oracle as O
from paper_2104_00359_gb300 import synthetic as S

from gpu_helpers import FIELDS, gpu_run

# The adjoint is held to 3e-4 of a gradient's scale at 8 bands; the pairs below
# keep |1 - r^2 / D^2| >= 1e-3, which float32 gives to 2^-24 / 1e-3 = 6e-5.
GATE = 1e-3
SPHERES = (1, 2, 7, 8, 9, 15, 16, 17, 31, 32, 33, 47, 63, 64, 65, 97)
SUMS = ("d_light", "d_centers", "d_radii", "d_points")


def _scene(n, spheres):
    """70 points (two 64-point tiles, three 32-point rows) away from the spheres' surfaces and centres."""
    sc = S.random_scene(7000 + 100 * n + spheres, 300, spheres, n, r_range=(0.03, 0.15))
    D = np.linalg.norm(sc["points"][:, None].astype(np.float64) - sc["centers"][None], axis=2)
    s2 = (sc["radii"] / D) ** 2
    keep = np.nonzero(np.all((np.abs(1 - s2) >= 1e-3) & (s2 < 16), axis=1))[0][:70]
    assert len(keep) == 70
    sc = dict(sc, **{k: np.ascontiguousarray(sc[k][keep]) for k in ("points", "normals", "albedo")})
    return sc, np.random.default_rng(spheres).normal(size=(70, 3)).astype(np.float32)


@pytest.mark.parametrize("n", range(1, 9))
def test_a_missing_sphere_would_show(n):
    """Every sphere's own sums are far above the gate (checked with the oracle
    alone); a sphere that hides the others wholly would not be."""
    for spheres in SPHERES[::3]:
        sc, dB = _scene(n, spheres)
        ref = O.shade_backward(O.Config(n_bands=n), *[sc[x] for x in FIELDS], dB)
        g = np.concatenate([ref["d_centers"], ref["d_radii"][:, None]], 1)
        a = np.concatenate([ref["abs_d_centers"], ref["abs_d_radii"][:, None]], 1)
        assert np.all(np.max(np.abs(g) / a, axis=1) > 5 * GATE)


@pytest.mark.gpu
@pytest.mark.parametrize("spheres", SPHERES)
@pytest.mark.parametrize("n", range(1, 9))
def test_sphere_groups_match_oracle(n, spheres):
    sc, dB = _scene(n, spheres)
    cfg = O.Config(n_bands=n)
    _, k, _, g, status = gpu_run(sc, cfg, dB=dB)
    assert status == 0
    ref = O.shade_backward(cfg, *[sc[x] for x in FIELDS], dB, k=k)
    for name in SUMS:
        assert np.all(np.abs(g[name].astype(np.float64) - ref[name]) <= GATE * ref["abs_" + name]), name

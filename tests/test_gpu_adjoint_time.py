"""Costs that must stay in proportion, each against another time of the same
run (no absolute figures): the adjoint's point gradients for few spheres, and
squarings whose number differs from point to point."""

import numpy as np
import pytest

from paper_2104_00359_gb300 import synthetic as S

from gpu_helpers import to_dev

pytestmark = pytest.mark.gpu


def _adjoint_us(n, points, spheres, want=None, fixed_k=-1):
    import torch
    from paper_2104_00359_gb300 import Config, Scene
    dev = torch.device("cuda:0")
    T = to_dev(S.random_scene(1, points, spheres, n), dev)
    scene = Scene(T["centers"], T["radii"], T["light"], Config(n_bands=n, fixed_k=fixed_k))
    saved = scene.new_saved(points, dev)
    args = (T["points"], T["normals"], T["albedo"])
    dB = torch.from_numpy(np.random.default_rng(0).normal(size=(points, 3)).astype(np.float32)).to(dev)
    scene.shade(*args, saved=saved)
    best = np.inf
    for _ in range(6):
        a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
        a.record()
        for _ in range(10):
            scene.backward(*args, dB, saved=saved, want=want or scene.ALL)
        b.record()
        torch.cuda.synchronize()
        best = min(best, a.elapsed_time(b) * 100.0)
    scene.close()
    return best


@pytest.mark.parametrize("n", [2, 3, 4])
def test_point_gradients_of_few_spheres(n):
    """With 20 spheres they cost little next to the spheres' own (a sum over the
    lanes per row of points made them 1.5 to 1.8 times the whole)."""
    sub = _adjoint_us(n, 1 << 18, 20, ("light", "albedo", "centers", "radii"))
    assert _adjoint_us(n, 1 << 18, 20) < 1.3 * sub


@pytest.mark.parametrize("n", [4, 5])
def test_squarings_that_differ_by_point(n):
    """1M points whose squarings number 0 to 4 against two for each (warps that
    drift apart in code larger than the instruction cache: 4 times at 5 bands)."""
    two = _adjoint_us(n, 1 << 20, 12, ("light", "albedo", "centers", "radii"), fixed_k=2)
    assert _adjoint_us(n, 1 << 20, 12, ("light", "albedo", "centers", "radii")) < 2.0 * two

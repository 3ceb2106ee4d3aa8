"""The batched L2 loss of many tiles: as exact as a sum of a million residuals
in float64, whatever order the tiles finish in."""

import ctypes

import pytest

from paper_2104_00359_gb300 import synthetic as S

from gpu_helpers import FIELDS

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [3, 6])
@pytest.mark.parametrize("points", [1, 1 << 20])
def test_batch_loss(n, points):
    """Each tile's total carries a few roundings of its own (2^-24 each, either
    way: nothing is left of them over 8,000 tiles, and 12 of them for one), the
    tiles' sum none, the result one: 2^-23, or 13 x 2^-24 for a single tile."""
    import torch
    from paper_2104_00359_gb300 import Config, Scene, _lib
    dev = torch.device("cuda:0")
    lib = _lib.load()
    sc = S.random_scene(33 + n, points, 3, n)
    T = {k: torch.from_numpy(sc[k]).to(dev) for k in FIELDS}
    target = torch.rand((points, 3), device=dev, generator=torch.Generator(dev).manual_seed(n))
    scene = Scene(T["centers"], T["radii"], T["light"], Config(n_bands=n))
    out = dict(radiance=torch.zeros((points, 3), device=dev), saved=scene.new_saved(points, dev),
               loss=torch.zeros((), device=dev))
    r = _lib.ShsRequest()
    r.scene, r.n_points, r.target = scene.handle.value, points, target.data_ptr()
    for k in ("points", "normals", "albedo"):
        setattr(r, k, T[k].data_ptr())
    for k, v in out.items():
        setattr(r, k, v.data_ptr())
    h = ctypes.c_void_p()
    _lib.check(lib.shs_batch_create(ctypes.byref(h)), "shs_batch_create")
    for _ in range(2):   # the accumulator is clean again for a second call
        _lib.check(lib.shs_shade_batch(h, (_lib.ShsRequest * 1)(r), 1, _lib.current_stream()), "shs_shade_batch")
        torch.cuda.synchronize()
        ref = 0.5 * float(((out["radiance"] - target).double() ** 2).sum())
        assert abs(float(out["loss"]) - ref) <= (13 * 2.0 ** -24 if points == 1 else 2.0 ** -23) * ref
    _lib.check(lib.shs_batch_destroy(h), "shs_batch_destroy")
    scene.close()

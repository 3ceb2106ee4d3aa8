"""A batch takes one launch per band count and pass, whatever mixture of horizon
culling and exponentials its requests ask for (small requests would each wait
for the others' launches otherwise)."""

import ctypes

import pytest

from paper_2104_00359_gb300 import synthetic as S

from gpu_helpers import to_dev

pytestmark = pytest.mark.gpu

MIXTURES = [[(0, 0)] * 3, [(1, 0), (0, 0)], [(0, 1), (0, 0)], [(1, 1), (0, 0), (0, 1), (1, 0)], [(0, 1), (1, 1)]]


@pytest.mark.parametrize("n", [4, 6, 7, 8])
@pytest.mark.parametrize("mixture", MIXTURES, ids=str)
def test_one_launch_per_pass(n, mixture):
    import torch
    from paper_2104_00359_gb300 import Config, Scene, _lib
    lib, dev = _lib.load(), torch.device("cuda:0")
    keep, reqs = [], []
    for i, (cull, mode) in enumerate(mixture):
        T = to_dev(S.random_scene(70 + i, 100, 9, n), dev)
        scene = Scene(T["centers"], T["radii"], T["light"], Config(n_bands=n, horizon_cull=bool(cull), exp_mode=mode))
        T.update(target=torch.zeros((100, 3), device=dev), radiance=torch.zeros((100, 3), device=dev),
                 saved=scene.new_saved(100, dev), d_light=torch.zeros((3, n * n), device=dev))
        r = _lib.ShsRequest()
        r.scene, r.n_points = scene.handle.value, 100
        for k in ("points", "normals", "albedo", "target", "radiance", "saved", "d_light"):
            setattr(r, k, T[k].data_ptr())
        keep.append((scene, T))
        reqs.append(r)
    h = ctypes.c_void_p()
    _lib.check(lib.shs_batch_create(ctypes.byref(h)), "shs_batch_create")
    before = lib.shs_launch_count()
    _lib.check(lib.shs_shade_batch(h, (_lib.ShsRequest * len(reqs))(*reqs), len(reqs), _lib.current_stream()),
               "shs_shade_batch")
    torch.cuda.synchronize()
    assert lib.shs_launch_count() - before == 2
    _lib.check(lib.shs_batch_destroy(h), "shs_batch_destroy")

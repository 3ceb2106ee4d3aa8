"""The adjoint kernels at the edges of their tiles: 6 to 8 bands (a lane pair
per point, 64-point tiles, 16 points per warp, 8 / 16 / 32 spheres per warp
step) and 1 to 5 bands; every variant of the batched kernels of 6 and more
bands against the single calls."""

import ctypes

import numpy as np
import pytest

from oracle import shs_oracle as O
from paper_2104_00359_gb300 import synthetic as S

from gpu_helpers import FIELDS, GRADS, gpu_run

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [6, 7, 8])
@pytest.mark.parametrize("points,spheres", [(1, 1), (15, 7), (16, 8), (17, 9), (63, 16), (64, 17), (65, 31), (127, 32),
                                            (129, 33), (70, 65)])
def test_tile_edges(n, points, spheres):
    """Points are independent: the per-point outputs of a call that ends inside
    a tile, warp or sphere group equal those of a larger call, bit for bit, and
    the scene-level sums of the call and of one on the other points add up to
    the larger call's: each term is the same number in both, so they differ by
    the rounding of three sums of at most 200 terms, 2 x 200 x 2^-24 of
    sum |terms| (the oracle's)."""
    total = 200
    full = S.random_scene(9000 + 100 * n + points, total, spheres, n, inside_fraction=0.05)
    dB = np.random.default_rng(points).normal(size=(total, 3)).astype(np.float32)
    cut = lambda a, b: dict(full, **{x: np.ascontiguousarray(full[x][a:b])   # noqa: E731
                                     for x in ("points", "normals", "albedo")})
    cfg = O.Config(n_bands=n)
    for saved in (True, False):
        B1, k1, f1, g1, s1 = gpu_run(full, cfg, dB=dB, saved=saved)
        B, k, f, g, s0 = gpu_run(cut(0, points), cfg, dB=dB[:points], saved=saved)
        rest = gpu_run(cut(points, total), cfg, dB=dB[points:], saved=saved)[3]
        assert s0 == 0 and s1 == 0
        for x, y in ((B, B1), (k, k1), (f, f1)) + tuple((g[m], g1[m]) for m in ("d_albedo", "d_points", "d_normals")):
            assert np.array_equal(x, y[:points])
        ref = O.shade_backward(cfg, *[full[x] for x in FIELDS], dB, k=k1)
        for name in ("d_light", "d_centers", "d_radii"):
            off = np.abs(g[name].astype(np.float64) + rest[name] - g1[name])
            assert np.all(off <= 2 * total * 2.0 ** -24 * ref["abs_" + name] + 1e-30), name


@pytest.mark.parametrize("n", [1, 2, 3, 4, 5])
@pytest.mark.parametrize("points,spheres", [(1, 1), (31, 8), (32, 9), (33, 17), (127, 31), (129, 32), (65, 33),
                                            (97, 64), (128, 71)])
def test_tile_edges_low_bands(n, points, spheres):
    """1 to 5 bands: two points per row of the pair adjoint, a lane pair per row
    from 32 spheres on, spheres on the lanes below."""
    test_tile_edges(n, points, spheres)


@pytest.mark.parametrize("n", [6, 8])
def test_batch_variants_match_single_calls(n):
    """One batch over the four kernel variants (horizon culling x projected
    exponential) and two sizes; float32 sums in another order only."""
    import torch
    from paper_2104_00359_gb300 import Config, Scene, _lib
    dev = torch.device("cuda:0")
    lib = _lib.load()
    jobs = []
    for i, (cull, mode, P, N) in enumerate([(0, 0, 130, 33), (1, 0, 64, 9), (0, 1, 65, 20), (1, 1, 200, 5),
                                            (0, 0, 1, 1), (1, 1, 63, 40)]):
        sc = S.random_scene(9900 + i, P, N, n)
        T = {k: torch.from_numpy(sc[k]).to(dev) for k in FIELDS}
        T["target"] = torch.rand((P, 3), device=dev, generator=torch.Generator(dev).manual_seed(i))
        cfg = Config(n_bands=n, horizon_cull=bool(cull), exp_mode=mode)
        single = Scene(T["centers"], T["radii"], T["light"], cfg)
        sv = single.new_saved(P, dev)
        B = single.shade(T["points"], T["normals"], T["albedo"], saved=sv)
        g = single.backward_l2(T["points"], T["normals"], T["albedo"], B, T["target"], saved=sv)
        batched = Scene(T["centers"], T["radii"], T["light"], cfg)
        out = dict(radiance=torch.zeros((P, 3), device=dev), saved=batched.new_saved(P, dev),
                   loss=torch.zeros((), device=dev), **batched._grad_buffers(P, dev, batched.ALL))
        r = _lib.ShsRequest()
        r.scene, r.n_points = batched.handle.value, P
        for k in ("points", "normals", "albedo", "target"):
            setattr(r, k, T[k].data_ptr())
        for k, v in out.items():
            setattr(r, k, v.data_ptr())
        jobs.append((r, B, g, out, (T, single, batched)))
    h = ctypes.c_void_p()
    _lib.check(lib.shs_batch_create(ctypes.byref(h)), "shs_batch_create")
    arr = (_lib.ShsRequest * len(jobs))(*[j[0] for j in jobs])
    for _ in range(2):   # the accumulators are clean again for a second call
        _lib.check(lib.shs_shade_batch(h, arr, len(jobs), ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)),
                   "shs_shade_batch")
        torch.cuda.synchronize()
        for r, B, g, out, _ in jobs:
            assert torch.equal(out["radiance"], B)
            for k in ("loss",) + GRADS:
                x, y = out[k].double(), g[k].double()
                assert (x - y).abs().max() <= 2e-6 * max(float(y.abs().max()), 1e-6), k
    _lib.check(lib.shs_batch_destroy(h), "shs_batch_destroy")

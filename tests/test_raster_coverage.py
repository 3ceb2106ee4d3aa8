"""Which triangle a pixel on an edge shows: the device's coverage pass against
its float32 restatement (oracle/raster_oracle.coverage_f32), bit for bit, on
meshes whose edges run through pixel centres."""

import numpy as np
import pytest

from oracle import raster_oracle as R
from paper_2104_00359_gb300 import synthetic as S


def _centre_mesh(n, seed, k=6):
    """k x k vertices on pixel centres of an n x n image (identity projection)."""
    rng = np.random.default_rng(seed)
    q = R.pixel_centres(n, n)
    at = np.linspace(0, n - 1, k).astype(int)
    r = np.clip(at[:, None] + rng.integers(-1, 2, (k, k)), 0, n - 1)
    c = np.clip(at[None, :] + rng.integers(-1, 2, (k, k)), 0, n - 1)
    v = np.concatenate([q[r, c].reshape(-1, 2), rng.uniform(-0.5, 0.5, (k * k, 1))], 1).astype(np.float32)
    i = np.arange((k - 1) * k).reshape(k - 1, k)[:, :-1].reshape(-1)
    faces = np.stack([np.stack([i, i + 1, i + k], 1), np.stack([i + 1, i + k + 1, i + k], 1)], 1).reshape(-1, 3)
    return v, faces


CENTRES = [(n, seed) for n in (9, 23, 37) for seed in range(3)]


# the other product fused; the row's form at every pixel
OTHERS = [lambda a, b, p, lead: R._area32(a, b, p), lambda a, b, p, lead: R._edge32(a, b, p, False)]


def test_rounding_decides_pixels_of_these_meshes():
    """Each other rounding of the edge function moves pixels here, and all of
    them agree with the float64 oracle but on edges."""
    moved = [0, 0]
    for n, seed in CENTRES:
        v, faces = _centre_mesh(n, seed)
        a, *others = (R.coverage_f32(v, faces, np.eye(4), n, n, edge) for edge in (None, *OTHERS))
        moved = [m + np.sum(a != b) for m, b in zip(moved, others)]
        _, ref = R.rasterize(v, faces, np.eye(4), np.zeros((len(v), 3)), n, n)
        for r, c in np.argwhere(np.any([m != ref for m in (a, *others)], axis=0)):
            d = []   # smallest edge function of a triangle in question
            for f in {m[r, c] for m in (a, *others, ref)} - {-1}:
                p = v[faces[f], :2].astype(np.float64)
                E = np.array(R._edges(p[0], p[1], p[2], R.pixel_centres(n, n)[r, c]))
                d.append(np.abs(E).min())
            assert min(d) < 1e-6   # float32 rounding of products of size 1
    assert min(moved) > 10, moved


def _device_map(v, faces, P, H, W):
    import torch
    from paper_2104_00359_gb300.raster import rasterize
    dev = torch.device("cuda:0")
    T = lambda x, t: torch.from_numpy(np.ascontiguousarray(x, t)).to(dev)
    _, fi = rasterize(T(v, np.float32), torch.ones((len(v), 3), device=dev), T(faces, np.int32), P, H, W)
    return fi.cpu().numpy().astype(np.int64)


@pytest.mark.gpu
@pytest.mark.parametrize("n,seed", CENTRES)
def test_pixels_on_edges(n, seed):
    v, faces = _centre_mesh(n, seed)
    assert np.array_equal(_device_map(v, faces, np.eye(4, dtype=np.float32), n, n),
                          R.coverage_f32(v, faces, np.eye(4), n, n))


@pytest.mark.gpu
@pytest.mark.parametrize("H,W", [(37, 61), (200, 301), (768, 768)])
def test_perspective_mesh(H, W):
    m = S.mesh_deformation_scene(seed=2, n_theta=120, n_phi=100, n_spheres=8, n_params=4, n_views=2)
    faces = S.uv_grid_faces(120, 100)
    P = S.look_at_perspective((2.5, 1.0, 1.2), aspect=W / H)
    assert np.array_equal(_device_map(m["v0"], faces, P, H, W), R.coverage_f32(m["v0"], faces, P, H, W))

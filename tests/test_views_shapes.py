"""ShadeViews forms each view's addresses itself: tensors that hold less than
the views read are refused before any launch, and larger ones are read at the
right places."""

import ctypes
from types import SimpleNamespace

import numpy as np
import pytest
import torch

from paper_2104_00359_gb300 import chain

V, P, N, NB = 3, 5, 2, 3


class _FakeLib:
    def __init__(self):
        self.calls, self.requests = [], []

    def shs_scenes_update(self, handles, n, centers, radii, light, stream):
        self.calls.append("update")
        self.centers = centers
        return 0

    def shs_shade_batch(self, batch, arr, n, stream):
        self.calls.append("shade")
        self.requests += [(r.points, r.normals, r.albedo) for r in arr]
        return 0


def _views(n_spheres=N):
    views = chain.ViewBatch.__new__(chain.ViewBatch)
    views.lib, views.V, views.P, views.N, views.K, views.batch = _FakeLib(), V, P, n_spheres, NB * NB, None
    views.scenes = [SimpleNamespace(handle=ctypes.c_void_p(i + 1), close=lambda: None) for i in range(V)]
    views.saved = [torch.empty(4) for _ in range(V)]
    return views


@pytest.fixture
def host(monkeypatch):
    """The host path without a GPU."""
    monkeypatch.setattr(chain, "_dev", lambda t, name: t.contiguous())
    monkeypatch.setattr(chain, "current_stream", lambda index=None: 0)


def _args(n_spheres=N, **shapes):
    s = dict(points=(V, P, 3), normals=(V, P, 3), albedo=(P, 3), centers=(V, n_spheres, 3), radii=(n_spheres,),
             light=(3, NB * NB))
    s.update(shapes)
    return [torch.zeros(v) for v in s.values()]


SHORT = [dict(points=(V - 1, P, 3)), dict(normals=(V - 1, P, 3)), dict(points=(V, P - 1, 3)),
         dict(normals=(V, P - 1, 3)), dict(albedo=(P - 1, 3)), dict(centers=(V - 1, N, 3)), dict(centers=(V, N - 1, 3)),
         dict(centers=(V, N + 1, 3)), dict(radii=(N - 1,)), dict(light=(3, NB)), dict(points=())]


@pytest.mark.parametrize("shapes", SHORT, ids=lambda s: "-".join(f"{k}{v}" for k, v in s.items()))
def test_short_tensors_are_refused(host, shapes):
    views = _views()
    with pytest.raises((ValueError, IndexError)):
        chain.ShadeViews.apply(*_args(**shapes), views)
    assert views.lib.calls == []


@pytest.mark.parametrize("shapes", [dict(points=(V - 1, P, 3)), dict(normals=(V - 1, P, 3)), dict(centers=(V - 1, 0, 3)),
                                    dict(albedo=(P - 1, 3))])
def test_short_tensors_are_refused_without_spheres(host, shapes):
    views = _views(0)
    with pytest.raises((ValueError, IndexError)):
        chain.ShadeViews.apply(*_args(0, **shapes), views)
    assert views.lib.calls == []


@pytest.mark.parametrize("shapes", [{}, dict(points=(V + 2, P, 3)), dict(normals=(V + 1, P, 3)),
                                    dict(centers=(V + 1, N, 3)), dict(points=(V, P + 4, 3), normals=(V, P + 2, 3)),
                                    dict(albedo=(P + 1, 3))])
def test_larger_tensors_are_read_in_place(host, shapes):
    views, args = _views(), _args(**shapes)
    chain.ShadeViews.apply(*args, views)
    assert views.lib.calls == ["update", "shade"]
    for v, (p, n, a) in enumerate(views.lib.requests):
        assert (p, n, a) == (args[0][v].data_ptr(), args[1][v].data_ptr(), args[2].data_ptr())


@pytest.mark.gpu
def test_larger_tensors_shade_the_same():
    """Views and points past the batch's are ignored."""
    from paper_2104_00359_gb300 import Config
    rng = np.random.default_rng(1)
    T = lambda *s: torch.from_numpy(rng.normal(size=s).astype(np.float32)).cuda()
    pts, nrm, alb = T(V + 1, P + 3, 3), T(V + 1, P + 3, 3), T(P + 3, 3)
    ctr, rad, light = 3.0 + T(V + 1, N, 3), torch.full((N,), 0.4).cuda(), T(3, NB * NB)
    views = chain.ViewBatch(V, P, ctr[0], rad, light, Config(n_bands=NB))
    big = chain.ShadeViews.apply(pts, nrm, alb, ctr, rad, light, views)
    fit = chain.ShadeViews.apply(pts[:V, :P].contiguous(), nrm[:V, :P].contiguous(), alb[:P], ctr[:V], rad, light, views)
    assert torch.equal(big, fit)
    views.close()

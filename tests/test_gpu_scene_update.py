"""Scene updates in one launch: shs_scenes_update of several scenes equals an
update of each, with any array left out, past one launch's 32 scenes."""

import ctypes

import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_scenes,N,bands", [(1, 5, 4), (3, 1, 1), (33, 200, 3), (16, 0, 2)])
@pytest.mark.parametrize("parts", ["crl", "c", "r", "l", "cl"])
def test_scenes_update_matches_single_updates(n_scenes, N, bands, parts):
    import torch
    from paper_2104_00359_gb300 import Config, Scene, _lib
    dev = torch.device("cuda:0")
    rnd = lambda *s: torch.rand(s, device=dev)   # noqa: E731
    cfg, K, P = Config(n_bands=bands), bands * bands, 70
    make = lambda: [Scene(rnd(N, 3) * 0 if N else None, rnd(N) * 0 + 0.1 if N else None,   # noqa: E731
                          torch.ones((3, K), device=dev), cfg) for _ in range(n_scenes)]
    one, many = make(), make()
    c, r, l = rnd(n_scenes, N, 3), rnd(N) * 0.2, rnd(3, K)
    for v, sc in enumerate(one):
        sc.update(centers=c[v] if "c" in parts else None, radii=r if "r" in parts else None,
                  light=l if "l" in parts else None)
    handles = (ctypes.c_void_p * n_scenes)(*[sc.handle.value for sc in many])
    lib = _lib.load()
    _lib.check(lib.shs_scenes_update(handles, n_scenes, c.data_ptr() if "c" in parts else None,
                                     r.data_ptr() if "r" in parts else None, l.data_ptr() if "l" in parts else None,
                                     _lib.current_stream()), "shs_scenes_update")
    pts, nrm, alb = rnd(P, 3) + 1.5, rnd(P, 3), rnd(P, 3)
    for x, y in zip(one, many):
        assert torch.equal(x.shade(pts, nrm, alb), y.shade(pts, nrm, alb))
    other = Scene(None, None, torch.ones((3, K + 2 * bands + 1), device=dev), Config(n_bands=bands + 1))
    bad = (ctypes.c_void_p * 2)(many[0].handle.value, other.handle.value)
    assert lib.shs_scenes_update(bad, 2, None, None, l.data_ptr(), _lib.current_stream()) == 1

"""rasterize() hands bare addresses to the kernels: tensors that are not on one
CUDA device are refused before anything is launched."""

import numpy as np
import pytest
import torch

from paper_2104_00359_gb300 import raster


class _Lib:
    """Stands in for the library: counts the launches."""

    def __init__(self):
        self.launches = 0

    def shs_raster_workspace_bytes(self, *a):
        return 1024

    def _launch(self, *a):
        self.launches += 1
        return 0

    shs_rasterize = shs_rasterize_backward = _launch


@pytest.fixture
def lib(monkeypatch):
    fake = _Lib()
    monkeypatch.setattr(raster._lib, "load", lambda: fake)
    monkeypatch.setattr(raster, "current_stream", lambda index=None: 0)
    return fake


def _mesh(device):
    v = torch.tensor([[-1.0, -1.0, 0.0], [1.0, -1.0, 0.0], [0.0, 1.0, 0.0]], device=device)
    return v, torch.ones((3, 3), device=device), torch.tensor([[0, 1, 2]], dtype=torch.int32, device=device)


@pytest.mark.parametrize("grad", [False, True])
def test_host_tensors_are_refused(lib, grad):
    v, b, f = _mesh("cpu")
    with pytest.raises(ValueError):
        raster.rasterize(v.requires_grad_(grad), b.requires_grad_(grad), f, np.eye(4), 4, 4)
    assert lib.launches == 0


class _Ctx:
    needs_input_grad = (True, True)
    size = (4, 4)
    P = np.eye(4, dtype=np.float32)

    def __init__(self, *saved):
        self.saved_tensors = saved


def test_host_gradient_is_refused(lib):
    v, b, f = _mesh("cpu")
    with pytest.raises(ValueError):
        raster.Rasterize.backward(_Ctx(v, b, f, torch.zeros((4, 4), dtype=torch.int32)), torch.zeros((4, 4, 3)), None)
    assert lib.launches == 0


@pytest.mark.gpu
@pytest.mark.parametrize("host", ["vertices", "radiance", "faces"])
def test_mixed_devices_are_refused(lib, host):
    t = dict(zip(("vertices", "radiance", "faces"), _mesh("cuda:0")))
    t[host] = t[host].cpu()
    with pytest.raises(ValueError):
        raster.rasterize(*t.values(), np.eye(4), 4, 4)
    assert lib.launches == 0

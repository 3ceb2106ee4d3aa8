"""The Legendre factors of the environment projection, bit for bit: of a map
that is zero but for one pixel of value 1, the m = 0 coefficients are
dOmega(row) N_l P_l(cos theta) without further rounding."""

import math

import numpy as np
import pytest

H, W, NB = 64, 4, 8
f32 = np.float32


def _restated(divide):
    """[H, NB] float32 restatement of the kernel's weights; divide: by l, or
    times its rounded reciprocal."""
    t = (np.arange(H) + 0.5) / H
    x, s = np.cos(math.pi * t).astype(f32), np.sin(math.pi * t).astype(f32)
    w = f32(2.0 * math.sin(math.pi / (2.0 * H)) * 2.0 * math.pi / W) * s
    P = [np.ones(H, f32), x]
    for l in range(2, NB):
        # one fused step, of which the product in float64 is exact to rounding's noise
        p = ((f32(2 * l - 1) * x).astype(np.float64) * P[-1] - (f32(l - 1) * P[-2]).astype(np.float64)).astype(f32)
        P.append(p / f32(l) if divide else p * (f32(1) / f32(l)))
    norm = [f32(math.sqrt((2 * l + 1) / (4 * math.pi))) for l in range(NB)]
    return np.stack([w * n * p for n, p in zip(norm, P)], 1)


@pytest.mark.gpu
def test_weights_divide_by_the_degree():
    """The device's sine and cosine may differ from the correctly rounded ones
    in places, so equality is asked of more entries than halfway between what
    the reciprocal form reaches and all."""
    import torch
    from paper_2104_00359_gb300.envmap import project_envmap
    env = torch.zeros((H, W, 3), device="cuda:0")
    got = np.zeros((H, NB), f32)
    for r in range(H):
        env.zero_()
        env[r, 0, 0] = 1.0
        light = project_envmap(env, NB).cpu().numpy()
        got[r] = [light[0, l * l + l] for l in range(NB)]
    ref, other = _restated(True)[:, 3:], _restated(False)[:, 3:]
    share = np.mean(ref == other)
    assert share < 0.9
    assert np.mean(got[:, 3:] == ref) > (1 + share) / 2, (np.mean(got[:, 3:] == ref), share)
    assert np.abs(got[:, 3:] - ref).max() < 1e-5 * np.abs(ref).max()

"""Weight gradients at the training size and on a grid of several tiles, where a
block keeps one fp32 sum over a range of z-planes: against fp64 sums of the
GPU's own bf16 operands (fp64 matrix products, one per tap).

Bound: a block adds about V / 152 voxels, 16 per step of its sum, and the blocks'
partials are added as 8 shares; with V = 2.8e5 that is at most 115 + 19 + 8
roundings of 2^-23 each: 1.7e-5 of the sum of the absolute terms, 2e-5 with the
products' own."""
import numpy as np
import pytest

from . import test_gpu_unet as U

pytestmark = pytest.mark.gpu


def _pool(x):
    import torch
    c, z, y, w = x.shape
    p = x.reshape(c, z // 2, 2, y // 2, 2, w // 2, 2).mean(dim=(2, 4, 6))
    return p.to(torch.bfloat16).double()


def _up(x):
    return x.repeat_interleave(2, 1).repeat_interleave(2, 2).repeat_interleave(2, 3)


def _wgrad(x, gz):
    """Weight gradient (cout, cin, 3, 3, 3) of a 3x3x3 'same' convolution."""
    import torch
    c, nz, ny, nx = x.shape
    xp = torch.nn.functional.pad(x, (1, 1, 1, 1, 1, 1))
    g = gz.reshape(gz.shape[0], -1)
    out = [g @ xp[:, dz:dz + nz, dy:dy + ny, dx:dx + nx].reshape(c, -1).T
           for dz in range(3) for dy in range(3) for dx in range(3)]
    return torch.stack(out, -1).reshape(gz.shape[0], c, 3, 3, 3)


@pytest.mark.parametrize("shape", [(64, 64, 64), (40, 60, 116)], ids=lambda s: "x".join(map(str, s)))
def test_weight_gradients_match_fp64_sums(shape):
    import torch

    import paper_2407_12399_gb300 as tsf
    f, g = U._inputs(shape, 2)
    net = U._net(U._params(5))
    A, G = net.debug(f, 0.05, g)
    _, grad = net.gradients(f, g, 0.05)
    got = tsf.unet_unflatten(grad)
    a = {k: torch.from_numpy(np.ascontiguousarray(v)).cuda().double() for k, v in A.items()}
    gz = {k: torch.from_numpy(np.ascontiguousarray(v)).cuda().double() for k, v in G.items()}
    inputs = {"e1a": a["x"], "e1b": a["e1a"], "e2a": _pool(a["e1b"]), "e2b": a["e2a"], "e3a": _pool(a["e2b"]),
              "e3b": a["e3a"], "d2a": torch.cat([_up(a["e3b"]), a["e2b"]]), "d2b": a["d2a"],
              "d1a": torch.cat([_up(a["d2b"]), a["e1b"]]), "d1b": a["d1a"]}
    for name, x in inputs.items():
        want, scale = _wgrad(x, gz[name]), _wgrad(x.abs(), gz[name].abs())
        diff = (torch.from_numpy(got[name + ".w"]).cuda().double() - want).abs()
        assert bool((diff <= 2e-5 * scale + 1e-30).all()), (name, float((diff / (scale + 1e-30)).max()))
        wb, sb = gz[name].sum(dim=(1, 2, 3)), gz[name].abs().sum(dim=(1, 2, 3))
        diff = (torch.from_numpy(got[name + ".b"]).cuda().double() - wb).abs()
        assert bool((diff <= 2e-5 * sb + 1e-30).all()), (name, float((diff / (sb + 1e-30)).max()))
    net.close()

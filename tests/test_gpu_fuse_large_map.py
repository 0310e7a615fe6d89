"""Fusion of a depth map of more than 2^31 pixels: the same as of a narrower
map (fewer pixels) that holds the same rows and columns where the voxels
project, bit for bit (the projections do not depend on the width)."""
import numpy as np
import pytest
import torch

import scenes
from scenes.configs import TsdfParams
from scenes.render import Pose, rot_xyz

pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_1809_06132_gb300 as P  # noqa: E402

X, Y = 100, 32780     # where the patch that is seen lies


def _run(width, height):
    cam = scenes.Camera(xi=1.0, fx=40.0, fy=40.0, cx=24.0 + X, cy=20.0 + Y, width=width, height=height)
    p = TsdfParams(voxel_size=0.1, mu=0.3, w_max=4.0, dense_dim=(16, 16, 16), origin=(-0.8, -0.8, 1.2))
    g = torch.Generator(device="cuda").manual_seed(6)
    vox = torch.rand((8, 512, 2), generator=g, device="cuda").requires_grad_()
    depth = torch.zeros((height, width), device="cuda")
    depth[Y:Y + 40, X:X + 48] = 1.6 + 0.3 * torch.rand((40, 48), generator=g, device="cuda")
    depth.requires_grad_()
    out = P.dense_fuse(vox, depth, p, cam, Pose(rot_xyz(0.01, 0.02, 0.0), np.array([0.02, -0.01, 0.03])))
    gv, gd = torch.autograd.grad(out.sum(), [vox, depth])
    return out.detach(), vox.detach(), gv, gd[Y:Y + 40, X:X + 48].clone(), gd.abs().sum(dtype=torch.float64)


def test_more_than_31_bits_of_pixels():
    if torch.cuda.mem_get_info()[0] < 40 << 30:
        pytest.skip("needs 40 GB of device memory")
    height = Y + 60
    assert 32768 * height < 2 ** 31 < 65536 * Y
    out, vox, gv, gd, s = _run(32768, height)
    OUT, VOX, GV, GD, S = _run(65536, height)
    assert torch.equal(vox, VOX) and (out != vox).any(-1).float().mean() > 0.3
    assert torch.equal(out, OUT) and torch.equal(gv, GV)
    assert (gd - GD).norm() <= 1e-5 * GD.norm() and abs(s - S) <= 1e-5 * S and S > 0

"""Differentiable fusion into a grid that starts anywhere in memory gives what
an aligned copy of it gives."""
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


@pytest.mark.parametrize("offset", [0, 1, 2, 3])
def test_grid_at_any_offset(offset):
    cam = scenes.Camera(xi=1.0, fx=40.0, fy=40.0, cx=24.0, cy=20.0, width=48, height=40)
    p = TsdfParams(voxel_size=0.1, mu=0.3, w_max=4.0, dense_dim=(16, 16, 8), origin=(-0.8, -0.8, 1.2))
    g = torch.Generator(device="cuda").manual_seed(5)
    flat = torch.rand(4 * 1024 + 4, generator=g, device="cuda")
    depth = 1.6 + 0.3 * torch.rand((40, 48), generator=g, device="cuda")
    up = torch.randn((4, 512, 2), generator=g, device="cuda")
    w2c = Pose(rot_xyz(0.01, 0.02, 0.0), np.array([0.02, -0.01, 0.03]))
    res = []
    for vox in (flat[offset:offset + 4096].view(4, 512, 2), flat[offset:offset + 4096].view(4, 512, 2).clone()):
        v, d = vox.detach().requires_grad_(), depth.clone().requires_grad_()
        out = P.dense_fuse(v, d, p, cam, w2c)
        res.append((out.detach(),) + torch.autograd.grad(out, [v, d], up))
    (o, gv, gd), (eo, egv, egd) = res
    assert torch.equal(o, eo) and torch.equal(gv, egv)
    # each pixel sums at most a few dozen FP32 terms in some order
    assert (gd - egd).abs().max() <= 64 * 2.0 ** -24 * egd.abs().max() and egd.any()
    if offset % 2:
        with pytest.raises(P.PsError):
            P.tsdf_integrate_dense_static(flat[offset:offset + 4096], p.dense_dim, p.origin, p.voxel_size, p.mu, p.w_max,
                                          depth, cam, w2c)

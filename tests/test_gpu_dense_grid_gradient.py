"""The gradient of a whole dense grid (pairs, cleared outputs) is that of the
separate form: D's gradients and the pose's bit for bit, the depth map's up
to the order of its atomic additions, zero for the weights; also for an
incoming gradient that starts between pairs in memory."""
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
from paper_1809_06132_gb300.psweep import tsdf_dense_fuse_backward  # noqa: E402


@pytest.mark.parametrize("dims,offset", [((8, 8, 8), 0), ((16, 24, 8), 1), ((40, 16, 32), 0)])
def test_grid_form_equals_the_separate_form(dims, offset):
    cam = scenes.Camera(xi=1.0, fx=40.0, fy=40.0, cx=24.0, cy=20.0, width=48, height=40)
    p = TsdfParams(voxel_size=0.1, mu=0.3, w_max=4.0, dense_dim=dims, origin=(-0.05 * dims[0], -0.05 * dims[1], 1.2))
    n = dims[0] * dims[1] * dims[2] // 512
    g = torch.Generator(device="cuda").manual_seed(3)
    vox = torch.rand((n, 512, 2), generator=g, device="cuda") * 2 - 1
    vox[..., 1] = torch.floor(5 * torch.rand((n, 512), generator=g, device="cuda"))
    depth = 1.6 + 0.5 * torch.rand((40, 48), generator=g, device="cuda")
    w2c = Pose(rot_xyz(0.01, 0.02, 0.0), np.array([0.02, -0.01, 0.03]))
    up = torch.randn(n * 1024 + 1, generator=g, device="cuda")[offset:offset + n * 1024].view(n, 512, 2)
    v, d = vox.requires_grad_(), depth.requires_grad_()
    delta = torch.zeros(6, dtype=torch.float64, requires_grad=True)
    out = P.dense_fuse(v, d, p, cam, w2c, delta)
    gv, gd, gp = torch.autograd.grad(out, [v, d, delta], up)
    ein, ed, ep = tsdf_dense_fuse_backward(vox.detach(), dims, p.origin, p.voxel_size, p.mu, p.w_max, depth.detach(), cam,
                                           w2c, up[..., 0])
    assert torch.equal(gv[..., 0], ein) and not gv[..., 1].any()
    assert torch.allclose(gp, ep.cpu(), rtol=1e-14, atol=0.0)
    # each pixel sums at most a few dozen FP32 terms in some order
    assert (gd - ed).abs().max() <= 64 * 2.0 ** -24 * ed.abs().max() and ed.any()

"""Dense fusion decides alike in both directions: the voxels whose value the
forward changes are those whose gradient the backward scales, and the pixel
that a voxel's value came from is the one its gradient goes to."""
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


@pytest.mark.parametrize("seed", range(4))
def test_forward_and_backward_observe_the_same(seed):
    rng = np.random.default_rng(seed)
    cam = scenes.Camera(xi=1.1, fx=150.0, fy=145.0, cx=81.3, cy=59.7, k1=-0.1, k2=0.02, p1=0.003, p2=-0.002, r2_max=2.0,
                        width=160, height=120)
    dims = (128, 96, 96)
    p = TsdfParams(voxel_size=0.02, mu=0.1, w_max=100.0, dense_dim=dims, origin=(-1.28, -0.96, 0.6))
    g = torch.Generator(device="cuda").manual_seed(seed)
    n = dims[0] * dims[1] * dims[2] // 512
    vox = torch.rand((n, 512, 2), generator=g, device="cuda") * 2 - 1
    vox[..., 1] = torch.floor(5 * torch.rand((n, 512), generator=g, device="cuda"))
    depth = 1.0 + 1.5 * torch.rand((120, 160), generator=g, device="cuda")
    depth[torch.rand((120, 160), generator=g, device="cuda") < 0.2] = 0.0
    w2c = Pose(rot_xyz(*rng.uniform(-0.1, 0.1, 3)), rng.uniform(-0.1, 0.1, 3))
    v, d = vox.clone().requires_grad_(), depth.clone().requires_grad_()
    out = P.dense_fuse(v, d, p, cam, w2c)
    one = torch.zeros_like(vox)
    one[..., 0] = 1.0
    gv, = torch.autograd.grad(out, [v], one, retain_graph=True)
    seen = out[..., 1] != vox[..., 1]
    assert torch.equal(seen, gv[..., 0] != 1.0) and 0.05 < seen.float().mean() < 0.95
    # every second pixel a little farther: the voxels that follow are those of these pixels
    board = (torch.arange(120, device="cuda")[:, None] + torch.arange(160, device="cuda")) % 2 == 1
    moved = P.dense_fuse(vox, depth + 0.01 * (board & (depth > 0)), p, cam, w2c)
    follow = seen & (moved[..., 1] != vox[..., 1]) & (moved[..., 0] != out[..., 0])
    gd, = torch.autograd.grad(out, [d], one * follow[..., None])
    assert not gd[~board].any() and (gd[board] > 0).float().mean() > 0.3

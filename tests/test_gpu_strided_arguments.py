"""Arguments that have to be copied before a kernel can read them (expanded
or strided gradients and blocks): each copy lives until the call has taken
its pointer, so that two of them never share an address."""
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


@pytest.mark.parametrize("w,h", [(96, 80), (61, 45)])
def test_expanded_gradients_of_a_soft_sweep(w, h):
    wl = scenes.diff(1, width=w, height=h, n_planes=8)
    imgs, _ = scenes.FrameSource(wl).frame(0)
    dev = [i.float().cuda() / 255.0 for i in imgs]
    sw = P.SoftSweep(wl.rig, wl.levels[0])
    _, _, aux = sw.forward(dev)
    one = torch.ones(1, device="cuda")
    gr, gc = (1.0 * one).expand(h, w), (-0.5 * one).expand(h, w)
    gi, gp = sw.backward(dev, None, aux, gr, gc)
    ei, ep = sw.backward(dev, None, aux, torch.full((h, w), 1.0, device="cuda"), torch.full((h, w), -0.5, device="cuda"))
    # the same kernel on the same values: only the order of its atomic additions differs
    for a, b in zip(gi + [gp], ei + [ep]):
        assert (a - b).norm() <= 1e-5 * b.norm() and b.any()
    # through autograd, from a plain weighted sum of both maps
    ims = [d.clone().requires_grad_() for d in dev]
    r, c = P.soft_depth(sw, ims)
    (r.sum() - 0.5 * c.sum()).backward()
    for a, b in zip(ims, ei):
        assert (a.grad - b).norm() <= 1e-5 * b.norm()


def test_strided_gradient_of_dense_fusion():
    cam = scenes.Camera(xi=1.0, fx=40.0, fy=40.0, cx=24.0, cy=20.0, width=48, height=40)
    p = TsdfParams(voxel_size=0.1, mu=0.3, w_max=4.0, dense_dim=(16, 16, 16), origin=(-0.8, -0.8, 1.2))
    g = torch.Generator(device="cuda").manual_seed(1)
    vox = torch.rand((8, 512, 2), generator=g, device="cuda")
    depth = 2.0 + 0.1 * torch.rand((40, 48), generator=g, device="cuda")
    up = torch.randn((8, 512, 2), generator=g, device="cuda")
    args = (vox, p.dense_dim, p.origin, p.voxel_size, p.mu, p.w_max, depth, cam,
            Pose(rot_xyz(0.01, 0.02, 0.0), np.array([0.02, -0.01, 0.03])))
    a, b = tsdf_dense_fuse_backward(*args, up[..., 0]), tsdf_dense_fuse_backward(*args, up[..., 0].contiguous())
    assert torch.equal(a[0], b[0]) and torch.allclose(a[1], b[1], rtol=1e-5, atol=1e-6) and b[1].any()


def test_strided_blocks_of_a_map():
    wl = scenes.diff(0)
    p = TsdfParams(voxel_size=0.1, mu=0.3, w_max=100.0, hash_slots=1 << 10, pool_blocks=64)
    n = 40
    g = torch.Generator(device="cuda").manual_seed(2)
    dw = torch.rand((n, 512, 2), generator=g, device="cuda")
    keys = torch.arange(3 * n, dtype=torch.int32, device="cuda").reshape(3, n).t()
    m = P.Tsdf(p, wl.rig.ref)
    m.load_blocks(keys, dw[..., 0], dw[..., 1])
    k, D, W = m.extract()
    order = torch.argsort(k[:, 0])
    assert torch.equal(k[order], keys) and torch.equal(D[order], dw[..., 0]) and torch.equal(W[order], dw[..., 1])


@pytest.mark.parametrize("foreign", [False, True])
def test_strided_gradients_on_another_stream(foreign):
    wl = scenes.diff(1, width=64, height=48, n_planes=8)
    imgs, _ = scenes.FrameSource(wl).frame(0)
    dev = [i.float().cuda() / 255.0 for i in imgs]
    sw = P.SoftSweep(wl.rig, wl.levels[0])
    r, c, aux = sw.forward(dev)
    g = torch.randn((64, 48), device="cuda")
    expect, _ = sw.backward(dev, None, aux, g.t().contiguous(), (2 * g).t().contiguous())
    side = torch.cuda.Stream()

    class Handle:           # what another library's stream looks like
        cuda_stream = side.cuda_stream
    for _ in range(3):
        torch.cuda.synchronize()
        got, _ = sw.backward(dev, None, aux, g.t(), (2 * g).t(), stream=Handle() if foreign else side)
        torch.cuda.synchronize()
        for a, b in zip(got, expect):
            assert (a - b).norm() <= 1e-5 * b.norm() and b.any()


def test_gradients_are_cleared_on_the_stream_of_the_call():
    # the current stream is busy: what is cleared there is cleared after the kernel has added to it
    wl = scenes.diff(1, width=64, height=48, n_planes=8)
    imgs, _ = scenes.FrameSource(wl).frame(0)
    dev = [i.float().cuda() / 255.0 for i in imgs]
    sw = P.SoftSweep(wl.rig, wl.levels[0])
    r, c, aux = sw.forward(dev)
    one = torch.ones_like(r)
    ei, ep = sw.backward(dev, None, aux, one, one)
    cam = scenes.Camera(xi=1.0, fx=40.0, fy=40.0, cx=24.0, cy=20.0, width=48, height=40)
    p = TsdfParams(voxel_size=0.1, mu=0.3, w_max=4.0, dense_dim=(16, 16, 16), origin=(-0.8, -0.8, 1.2))
    args = (torch.rand((8, 512, 2), device="cuda"), p.dense_dim, p.origin, p.voxel_size, p.mu, p.w_max,
            2.0 + 0.1 * torch.rand((40, 48), device="cuda"), cam, Pose(rot_xyz(0.01, 0.02, 0.0), np.array([0.02, -0.01, 0.03])),
            torch.randn((8, 512), device="cuda"))
    expect = ei + [ep] + list(tsdf_dense_fuse_backward(*args))
    side = torch.cuda.Stream()
    torch.cuda.synchronize()
    torch.cuda._sleep(200_000_000)          # about 0.1 s
    gi, gp = sw.backward(dev, None, aux, one, one, stream=side)
    got = gi + [gp] + list(tsdf_dense_fuse_backward(*args, stream=side))
    torch.cuda.synchronize()
    for a, b in zip(got, expect):
        assert (a - b).norm() <= 1e-5 * b.norm() and b.any()

"""The image gradients of a soft sweep are tensors of their own: each holds
its own memory and version, and takes every in-place operation."""
import pytest
import torch

import scenes

pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_1809_06132_gb300 as P  # noqa: E402


def test_gradients_are_independent_tensors():
    wl = scenes.diff(2, width=48, height=40, n_planes=4)
    imgs, _ = scenes.FrameSource(wl).frame(0)
    ims = [(i.float().cuda() / 255.0).requires_grad_() for i in imgs]
    sw = P.SoftSweep(wl.rig, wl.levels[0])
    r, c = P.soft_depth(sw, ims)
    grads = torch.autograd.grad(r.sum() + c.sum(), ims)
    assert len({g.untyped_storage().data_ptr() for g in grads}) == len(grads)
    for g, im in zip(grads, ims):
        assert g.shape == im.shape and g.any() and not g._is_view()
        assert g.untyped_storage().nbytes() < 2 * g.numel() * 4
    before = [g._version for g in grads]
    x = torch.ones((), device="cuda", requires_grad=True)
    grads[1].detach_()
    grads[1].mul_(x)       # in place with a tensor that requires gradients
    assert grads[1].requires_grad and [g._version for g in grads[2:]] == before[2:] and grads[0]._version == before[0]

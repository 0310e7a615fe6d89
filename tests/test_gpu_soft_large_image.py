"""Soft sweep with a matching image of more than 2^31 texels: the same as with
a narrower image (fewer texels) that holds the same rows and columns where
the samples fall, bit for bit (the projections do not depend on the width)."""
import dataclasses

import pytest
import torch

import scenes

pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_1809_06132_gb300 as P  # noqa: E402

W, H, X, Y = 64, 48, 100, 32780     # the patch that is seen, and where it lies


def _run(wl, patch, width, height):
    cam = wl.rig.cams[0]
    cam = dataclasses.replace(cam, width=width, height=height, cx=cam.cx + X, cy=cam.cy + Y)
    rig = dataclasses.replace(wl.rig, cams=[cam], ref_to_cam=wl.rig.ref_to_cam[:1])
    big = torch.zeros((height, width), device="cuda")
    big[Y:Y + H, X:X + W] = patch[1]
    sw = P.SoftSweep(rig, wl.levels[0])
    r, c, aux = sw.forward([patch[0], big])
    gi, gp = sw.backward([patch[0], big], None, aux, torch.ones_like(r), torch.ones_like(c))
    return r, c, gi[0], gi[1][Y - 1:Y + H + 1, X - 1:X + W + 1].clone(), gi[1].abs().sum(dtype=torch.float64), gp


def test_more_than_31_bits_of_texels():
    if torch.cuda.mem_get_info()[0] < 40 << 30:
        pytest.skip("needs 40 GB of device memory")
    wl = scenes.diff(6, width=W, height=H, n_planes=6)
    imgs, _ = scenes.FrameSource(wl).frame(0)
    patch = [i.float().cuda() / 255.0 for i in imgs[:2]]
    height = Y + H + 20
    assert 32768 * height < 2 ** 31 < 65536 * Y
    r, c, g0, g1, s, gp = _run(wl, patch, 32768, height)
    R, C, G0, G1, S, GP = _run(wl, patch, 65536, height)
    assert (r > 0).float().mean() > 0.3
    assert torch.equal(r, R) and torch.equal(c, C)
    # (atomic additions in any order)
    for a, b in ((g0, G0), (g1, G1), (gp, GP)):
        assert b.any() and (a - b).norm() <= 1e-5 * b.norm()
    assert abs(s - S) <= 1e-5 * S and S > 0

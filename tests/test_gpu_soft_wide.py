"""Soft sweep of images large enough for the forward's wide tiles (at least as
many tiles of 32 x 16 pixels as the GPU has SMs; remainders in both
directions), for every window: bit for bit what the small tiles give on a
strip of the image, and against the FP64 oracle within the bounds of the other
soft-sweep tests.  And the backward's layouts (window x cameras) that those
tests leave out, at their size and within their bounds."""
import dataclasses
import math

import numpy as np
import pytest
import torch

import oracle
import scenes
from scenes.render import Pose, rot_xyz

pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_1809_06132_gb300 as P  # noqa: E402

W, H = 417, 193


def _case(seed, w, h, window, n_cams, n_planes):
    wl = scenes.diff(seed, width=w, height=h, n_planes=n_planes)
    cams, poses = list(wl.rig.cams), list(wl.rig.ref_to_cam)
    for k, dy in enumerate((-0.3, 0.3)):
        R = rot_xyz(math.radians(0.5 * (k + 1)), math.radians(-0.4), 0.0)
        poses.append(Pose(R.T, -R.T @ np.array([0.1, dy, 0.0])))
        cams.append(cams[k])
    lv = dataclasses.replace(wl.levels[0], window=window)
    wl.rig = dataclasses.replace(wl.rig, cams=cams[:n_cams], ref_to_cam=poses[:n_cams])
    imgs, _ = scenes.FrameSource(wl).frame(0)
    dev = [torch.from_numpy((i.numpy().astype(np.float64) / 255.0).astype(np.float32)).cuda() for i in imgs]
    return wl.rig, lv, dev, [d.double().cpu().numpy() for d in dev]


@pytest.mark.parametrize("window,n_cams,n_planes", [(5, 1, 19), (5, 2, 34), (5, 3, 7), (5, 4, 1), (7, 2, 17), (7, 4, 5),
                                                    (9, 1, 18), (9, 2, 5), (9, 4, 3)])
def test_wide_tiles(window, n_cams, n_planes):
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    assert -(-W // 32) * -(-H // 16) >= sms > -(-W // 32) * -(-64 // 16)
    rig, lv, dev, ims = _case(8, W, H, window, n_cams, n_planes)
    sw = P.SoftSweep(rig, lv, temperature=0.05)
    r, S, aux = sw.forward(dev)

    # a strip of the reference image has few tiles, so the small ones
    y0, h, rho = 71, 64, window // 2
    ref = dataclasses.replace(rig.ref, height=h, cy=rig.ref.cy - y0)
    strip = P.SoftSweep(dataclasses.replace(rig, ref=ref), lv, temperature=0.05)
    sr, sS, saux = strip.forward([dev[0][y0:y0 + h].contiguous()] + dev[1:])
    for a, b in ((r, sr), (S, sS), (aux, saux)):
        assert torch.equal(a[y0 + rho:y0 + h - rho], b[rho:h - rho])

    orr, oS = oracle.soft_depth(rig, lv, ims, T=0.05, with_cost=True)
    rc, Sc = r.cpu().numpy(), S.cpu().numpy()
    both = (rc > 0) & (orr > 0)
    assert both.mean() > 0.3 and ((rc > 0) == (orr > 0)).mean() >= 0.99
    assert np.median(np.abs(rc[both] - orr[both]) / orr[both]) <= 1e-5
    assert (np.abs(Sc[both] - oS[both]) <= 1e-4).mean() >= 0.995


@pytest.mark.parametrize("window,n_cams", [(5, 1), (5, 3), (5, 4), (7, 1), (7, 2), (7, 4), (9, 1), (9, 2), (9, 3)])
def test_backward_layouts(window, n_cams):
    rig, lv, dev, ims = _case(5, 64, 48, window, n_cams, 8)
    sw = P.SoftSweep(rig, lv, temperature=0.05)
    r, _, aux = sw.forward(dev)
    valid = (r.cpu().numpy() > 0) & ~oracle.soft_depth_ties(rig, lv, ims, tau=1e-5, tau_px=3e-5)
    assert valid.mean() > 0.3
    rng = np.random.default_rng(2)
    g = (rng.normal(size=valid.shape) * valid).astype(np.float32)
    gs = (rng.normal(size=valid.shape) * valid).astype(np.float32)
    gi, gp = sw.backward(dev, None, aux, torch.from_numpy(g).cuda(), torch.from_numpy(gs).cuda())
    ogi, ogp = oracle.soft_depth_grad(rig, lv, ims, g.astype(np.float64), T=0.05, g_cost=gs.astype(np.float64))
    compared = 0
    for a, b in zip([x.cpu().numpy() for x in gi] + list(gp.cpu().numpy()), list(ogi) + list(ogp)):
        assert np.isfinite(a).all()
        if np.abs(b).max() > 0:
            assert np.linalg.norm(a - b) <= 1e-4 * np.linalg.norm(b)
            compared += 1
    assert compared >= 3

"""Soft sweep at the edges of its tiling (32 x 16 and 16 x 16 output tiles,
plane pairs, rounds of 16 planes shared by two groups of threads): forward maps and
gradients against the FP64 oracle, within the bounds the other soft-sweep
tests use."""
import numpy as np
import pytest
import torch

import oracle
import scenes

pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_1809_06132_gb300 as P  # noqa: E402


@pytest.mark.parametrize("w,h,planes", [(32, 16, 16), (33, 17, 17), (31, 47, 1), (48, 33, 130), (65, 16, 34)])
def test_tiles_and_plane_splits(w, h, planes):
    wl = scenes.diff(7, width=w, height=h, n_planes=planes)
    imgs, _ = scenes.FrameSource(wl).frame(0)
    dev = [torch.from_numpy((i.numpy().astype(np.float64) / 255.0).astype(np.float32)).cuda() for i in imgs]
    ims = [d.double().cpu().numpy() for d in dev]
    sw = P.SoftSweep(wl.rig, wl.levels[0], temperature=0.05)
    r, S, aux = sw.forward(dev)
    orr, oS = oracle.soft_depth(wl.rig, wl.levels[0], ims, T=0.05, with_cost=True)
    rc, Sc = r.cpu().numpy(), S.cpu().numpy()
    both = (rc > 0) & (orr > 0)
    assert ((rc > 0) == (orr > 0)).mean() >= 0.99
    if both.any():
        assert np.median(np.abs(rc[both] - orr[both]) / orr[both]) <= 1e-5
        assert (np.abs(Sc[both] - oS[both]) <= 1e-4).mean() >= 0.995
    tied = oracle.soft_depth_ties(wl.rig, wl.levels[0], ims, tau=1e-5, tau_px=3e-5)
    valid = (rc > 0) & ~tied
    rng = np.random.default_rng(3)
    g = (rng.normal(size=valid.shape) * valid).astype(np.float32)
    gs = (rng.normal(size=valid.shape) * valid).astype(np.float32)
    gi, gp = sw.backward(dev, None, aux, torch.from_numpy(g).cuda(), torch.from_numpy(gs).cuda())
    ogi, ogp = oracle.soft_depth_grad(wl.rig, wl.levels[0], ims, g.astype(np.float64), T=0.05,
                                      g_cost=gs.astype(np.float64))
    for a, b in zip([x.cpu().numpy() for x in gi] + list(gp.cpu().numpy()), list(ogi) + list(ogp)):
        assert np.isfinite(a).all()
        if np.abs(b).max() > 0:
            assert np.linalg.norm(a - b) <= 1e-4 * np.linalg.norm(b)

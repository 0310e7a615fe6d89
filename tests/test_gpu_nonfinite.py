"""Values at the ends of FP32, and what they may and may not reach."""
import dataclasses

import pytest
import torch

import scenes

pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_1809_06132_gb300 as P  # noqa: E402


@pytest.mark.parametrize("window", [5, 9])
def test_a_reference_pixel_that_is_no_number(window):
    wl = scenes.diff(3, width=64, height=48, n_planes=6)
    lv = dataclasses.replace(wl.levels[0], window=window)
    imgs, _ = scenes.FrameSource(wl).frame(0)
    dev = [i.float().cuda() / 255.0 for i in imgs]
    x, y = 37, 30            # not a tile's centre, whose value all of a tile is taken relative to
    dev[0][y, x] = float("nan")
    sw = P.SoftSweep(wl.rig, lv)
    r, c, aux = sw.forward(dev)
    gi, _ = sw.backward(dev, None, aux, torch.ones_like(r), torch.ones_like(c))
    rho = window // 2
    assert torch.isfinite(r).all() and not r[y - rho:y + rho + 1, x - rho:x + rho + 1].any()
    bad = ~torch.isfinite(gi[0])
    bad[y, x] = False        # (its own gradient has no value)
    assert not bad.any() and gi[0].nan_to_num().any()

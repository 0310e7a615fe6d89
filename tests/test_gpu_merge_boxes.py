"""Boxes of the merge are gathered per tile of output pixels: the masked map is
the unmasked one with every box's pixels zero, for boxes that end on tile
borders, lie outside the image, are empty, or are as many as a call may pass;
with and without the depth filters, whose launch merges and filters at once."""
import numpy as np
import pytest
import torch

import scenes

pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_1809_06132_gb300 as P  # noqa: E402


@pytest.mark.parametrize("window", [0, 1, 5, 15])   # 0: filters off
@pytest.mark.parametrize("n", [1, 16, 17, 256])
def test_boxes_mask_the_merged_map(window, n):
    wl = scenes.street(1, n_frames=1, scale=0.25)
    H, W = wl.rig.ref.height, wl.rig.ref.width
    ims = [i.cuda() for i in scenes.FrameSource(wl).frame(0)[0]]
    f = scenes.Filters(window=window, delta=0.1) if window else None
    sw = P.Sweep(wl.rig, wl.levels, filters=f)
    plain = sw.depth(ims)
    g = np.random.default_rng(n)
    b = np.empty((n, 4), np.int32)
    b[:, :2] = g.integers((-20, -20), (W, H), (n, 2))
    b[:, 2:] = b[:, :2] + g.integers(0, 24, (n, 2))
    b[0] = (32, 16, 64, 32)
    if n > 1:
        b[1], b[-1] = (31, 15, 33, 17), (W - 1, H - 1, W + 9, H + 9)
    keep = np.ones((H, W), bool)
    for x0, y0, x1, y1 in b:
        keep[max(y0, 0):max(y1, 0), max(x0, 0):max(x1, 0)] = False
    want = torch.where(torch.from_numpy(keep).cuda(), plain, torch.zeros_like(plain))
    assert torch.equal(sw.depth(ims, boxes=b), want)
    # a window of one pixel has no neighbours to agree with: it keeps nothing
    assert (plain > 0).sum() > 500 if window != 1 else not plain.any()

"""A batch made later does not change what an earlier one can launch: both
share a kernel, whatever shared memory each of them needs."""
import dataclasses

import pytest
import torch

import scenes

pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_1809_06132_gb300 as P  # noqa: E402


@pytest.mark.parametrize("use_graph", [False, True])
def test_a_smaller_batch_made_later(use_graph):
    wl = scenes.tiny(0)
    imgs, _ = scenes.FrameSource(wl).frame(0)
    dev = [i.cuda() for i in imgs]
    made = []
    for window in (9, 5):
        lv = [dataclasses.replace(wl.levels[0], window=window)]
        rig = wl.rig
        if window == 9:     # the wider window, and every camera twice: more shared memory
            rig = dataclasses.replace(rig, cams=rig.cams * 2, ref_to_cam=rig.ref_to_cam * 2)
        sw = P.Sweep(rig, lv)
        ims = [dev[0]] + dev[1:] * (len(rig.cams) // len(wl.rig.cams))
        made.append((sw, ims, P.Batch([sw], use_graph=use_graph)))
    for sw, ims, b in made:
        torch.cuda.synchronize()
        stream = torch.cuda.Stream()   # (a graph replay needs one of its own)
        out, = b.run([ims], stream=stream)
        stream.synchronize()
        assert b.status() == P.PS_OK
        assert torch.equal(out, sw.depth(ims)) and (out > 0).any()

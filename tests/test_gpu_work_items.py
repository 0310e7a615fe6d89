"""The split of a sweep into work items (planes per item) follows image size,
plane and camera count; the results do not: level outputs and depth are bit
for bit those of one work item per tile (a batch of one sweep with chunks of
all planes), from images of a few tiles to several waves of items, plane
counts that leave a short last item, and one and two levels."""
import dataclasses

import pytest
import torch

import scenes
from scenes.configs import CROP, DOWNSAMPLE, FRONTO, GROUND, Level, PlaneSet

pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_1809_06132_gb300 as P  # noqa: E402


@pytest.mark.parametrize("w,h,cams,planes,ground,crop", [
    (65, 25, 1, 1, 0, None), (160, 128, 1, 33, 0, None), (96, 72, 3, 130, 0, None), (320, 256, 2, 64, 32, (162, 130, 47)),
    (640, 480, 4, 65, 0, None)])
def test_results_do_not_depend_on_the_split(w, h, cams, planes, ground, crop):
    wl = scenes.batch_mix(5, n=1, sizes=((w, h),), planes=(32,), max_cams=1)[0]
    rig = wl.rig
    poses = [rig.ref_to_cam[0]] * cams
    rig = dataclasses.replace(rig, cams=[rig.cams[0]] * cams,
                              ref_to_cam=[dataclasses.replace(p, t=p.t * (1.0 + 0.2 * j)) for j, p in enumerate(poses)])
    sets = [PlaneSet(FRONTO, planes, 0.5, 30.0)]
    if ground:
        sets.append(PlaneSet(GROUND, ground, 1.1, 2.1, n=(0.0, 1.0, 0.0)))
    levels = [Level(kind=DOWNSAMPLE, factor=2 if crop else 1, window=7, sets=sets)]
    if crop:
        levels.append(Level(kind=CROP, window=9, crop_w=crop[0], crop_h=crop[1], sets=[PlaneSet(FRONTO, crop[2], 1.0, 80.0)]))
    ims = [i.cuda() for i in scenes.FrameSource(dataclasses.replace(wl, rig=rig, levels=levels)).frame(0)[0]]
    a, b = P.Sweep(rig, levels), P.Sweep(rig, levels)
    outs = a.alloc_level_outputs()
    da = a.depth(ims, level_outs=outs)
    db = P.Batch([b], plane_chunk=4096).run([ims])[0]
    for x, y in zip(outs, b.level_outputs()):
        for k in ("depth", "c1", "c2", "kstar"):
            assert torch.equal(x[k], y[k]), k
    assert torch.equal(da, db) and (da > 0).any()

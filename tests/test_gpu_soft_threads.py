"""Soft sweeps of several threads at once: handles of one window and different
numbers of cameras share kernels, but no launch depends on another's size."""
import dataclasses
import threading

import pytest
import torch

import scenes

pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_1809_06132_gb300 as P  # noqa: E402


@pytest.mark.parametrize("counts", [(1, 2, 1, 2), (3, 4, 3, 4)])
def test_handles_of_different_sizes_in_threads(counts):
    wl = scenes.diff(4, width=24, height=20, n_planes=2)
    lv = dataclasses.replace(wl.levels[0], window=9)
    imgs, _ = scenes.FrameSource(wl).frame(0)
    dev = [i.float().cuda() / 255.0 for i in imgs]
    L = P.load()
    work = []
    for n in counts:
        rig = dataclasses.replace(wl.rig, cams=(wl.rig.cams * 2)[:n], ref_to_cam=(wl.rig.ref_to_cam * 2)[:n])
        sw, ims = P.SoftSweep(rig, lv), [dev[0]] + (dev[1:] * 2)[:n]
        r, c, aux = sw.forward(ims)
        gi, gp = sw.backward(ims, None, aux, r, c)
        stream = torch.cuda.Stream()
        # the calls themselves, so that the threads spend their time in the library
        ptrs, poses = sw._args(ims, None)
        out = [torch.empty_like(t) for t in (r, c, aux)]
        work.append(dict(sw=sw, ims=ims, ptrs=ptrs, poses=poses, out=out, expect=(r, c, aux), stream=stream, gp=gp,
                         o=[t.data_ptr() for t in out]))
    torch.cuda.synchronize()
    bad = []

    def loop(w):
        s = w["stream"].cuda_stream
        for k in range(4000):
            st = L.psdiff_forward(w["sw"].h, w["ptrs"], w["poses"], *w["o"], s)
            if st == P.PS_OK:
                st = L.psdiff_backward(w["sw"].h, w["ptrs"], w["poses"], w["o"][2], w["o"][0], w["o"][1], None,
                                       w["gp"].data_ptr(), s)
            if st != P.PS_OK:
                bad.append((st, L.ps_last_error()))
                return
            if k % 100 == 0:
                w["stream"].synchronize()
        w["stream"].synchronize()

    threads = [threading.Thread(target=loop, args=(w,)) for w in work]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not bad
    for w in work:
        assert all(torch.equal(a, b) for a, b in zip(w["out"], w["expect"]))

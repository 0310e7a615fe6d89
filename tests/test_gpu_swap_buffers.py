"""tsdf_swap_out writes value pairs with 8-byte stores where the caller's
buffers allow it and single floats where they do not: both give the same
blocks, with room for all of them, for some, and for none."""
import ctypes as C

import numpy as np
import pytest
import torch

import scenes

pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_1809_06132_gb300 as P  # noqa: E402


@pytest.mark.parametrize("offset", [0, 1])   # floats by which the voxel buffers are off an 8-byte boundary
def test_swap_out_to_any_alignment(offset):
    wl = scenes.street(2, n_frames=1, scale=0.25)
    _, rng = scenes.FrameSource(wl).frame(0, with_range=True)
    depth = torch.from_numpy(rng.numpy().astype(np.float32)).cuda()
    far = (C.c_double * 3)(1e4, 0.0, 0.0)
    maps = [P.Tsdf(wl.tsdf, wl.rig.ref) for _ in range(2)]
    for m in maps:
        m.integrate(depth, wl.world_to_ref[0], wl.local_center(0))
    keys, D, W = maps[0].extract()
    want = {tuple(k): (d, w) for k, d, w in zip(keys.cpu().tolist(), D.cpu().numpy(), W.cpu().numpy())}
    n, got = len(want), {}
    assert n > 64 and any(w.any() for _, w in want.values())
    for cap in (0, 33, n):
        k = torch.full((n, 3), -7, dtype=torch.int32, device="cuda")
        d, w = (torch.full((n * 512 + 1,), -7.0, device="cuda") for _ in range(2))
        m = C.c_int64()
        st = P.load().tsdf_swap_out(maps[1].h, far, k.data_ptr(), d.data_ptr() + 4 * offset, w.data_ptr() + 4 * offset, cap,
                                    C.byref(m), None)
        left = n - len(got)
        assert st == (P.PS_OK if cap >= left else P.PS_ERR_CAPACITY) and m.value == min(cap, left)
        assert (k[m.value:] == -7).all() and (d[offset + 512 * m.value:] == -7.0).all()
        d, w = (t[offset:offset + 512 * m.value].cpu().numpy().reshape(-1, 512) for t in (d, w))
        for key, x, y in zip(k[:m.value].cpu().tolist(), d, w):
            assert tuple(key) not in got
            got[tuple(key)] = (x, y)
    assert maps[1].count() == 0 and got.keys() == want.keys()
    for key, (x, y) in got.items():   # extract zeroes D where nothing was observed, as the map does
        assert np.array_equal(y, want[key][1]) and np.array_equal(x, want[key][0])

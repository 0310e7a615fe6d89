"""Values at the ends of FP32, and what they may and may not reach."""
import dataclasses

import numpy as np
import pytest
import torch

import scenes
from scenes.configs import TsdfParams
from scenes.render import Pose

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


def _far_map(local_half):
    cam = scenes.Camera(xi=1.0, fx=40.0, fy=40.0, cx=24.0, cy=20.0, width=48, height=40)
    p = TsdfParams(voxel_size=0.02, mu=0.1, w_max=100.0, hash_slots=1 << 16, pool_blocks=1 << 14, local_half=local_half)
    # the optical axis along (1, 1, 1): every coordinate of the far point overflows a block count
    z = np.ones(3) / np.sqrt(3.0)
    x = np.array([1.0, -1.0, 0.0]) / np.sqrt(2.0)
    pose = Pose(np.stack([x, np.cross(z, x), z]), np.zeros(3))
    depth = torch.zeros((40, 48), device="cuda")
    depth[20, 24] = 2e38
    return P.Tsdf(p, cam), depth, pose


def test_a_range_beyond_the_largest_block_count():
    m, depth, pose = _far_map((3.0, 3.0, 3.0))
    m.integrate(depth, pose, (0.0, 0.0, 0.0))
    assert m.status() == P.PS_OK and m.count() == 0    # outside the local map: skipped
    m, depth, pose = _far_map(None)
    m.integrate(depth, pose)
    assert m.status() == P.PS_ERR_CAPACITY and m.count() == 0    # no local map: no key holds such a block


def test_variances_whose_product_overflows():
    # a correlation over an infinite deviation is 0: every such plane costs 1/2
    T = 0.05
    wl = scenes.diff(5, width=64, height=48, n_planes=6)
    imgs, _ = scenes.FrameSource(wl).frame(0)
    dev = [i.float().cuda() / 255.0 for i in imgs]
    sw = P.SoftSweep(wl.rig, wl.levels[0], temperature=T)
    usual, _, _ = sw.forward(dev)
    big = [1e12 * d for d in dev]
    r, c, aux = sw.forward(big)
    gi, gp = sw.backward(big, None, aux, torch.ones_like(r), torch.ones_like(c))
    assert (r > 0)[usual > 0].all() and torch.isfinite(r).all() and torch.isfinite(c).all()
    # the soft minimum of n equal costs is 1/2 - T log n: exp((1/2 - c) / T) is n, to the rounding of c over T
    n = torch.exp((0.5 - c[usual > 0]) / T)
    assert ((n - n.round()).abs() <= n * 2.0 ** -22 / T).all() and (n.round() >= 1).all() and (n.round() <= 6).all()
    assert all((g == 0).all() for g in gi) and (gp == 0).all()


@pytest.mark.parametrize("T", [1e-39, 1e-42])
def test_a_temperature_below_the_smallest_normal_number(T):
    # costs differ by 2^-25 or more: any such temperature takes the plane of the lowest cost alone
    wl = scenes.diff(5, width=48, height=40, n_planes=6)
    imgs, _ = scenes.FrameSource(wl).frame(0)
    dev = [i.float().cuda() / 255.0 for i in imgs]
    a, b = (P.SoftSweep(wl.rig, wl.levels[0], temperature=t).forward(dev) for t in (T, 1e-30))
    assert torch.equal(a[0], b[0]) and torch.equal(a[1], b[1]) and (a[0] > 0).any()


@pytest.mark.parametrize("value", [float("nan"), float("inf"), float("-inf")])
@pytest.mark.parametrize("window,x,y", [(5, 8, 8), (9, 24, 24), (7, 24, 8)])
def test_a_tile_centre_that_is_no_number(window, x, y, value):
    # the pixel that a tile's intensities are taken relative to, in tiles whose halo leaves the image:
    # nothing is written outside the image's gradient, and inside only its own value is none
    w = h = 32
    wl = scenes.diff(3, width=w, height=h, n_planes=6)
    lv = dataclasses.replace(wl.levels[0], window=window)
    imgs, _ = scenes.FrameSource(wl).frame(0)
    dev = [i.float().cuda() / 255.0 for i in imgs]
    dev[0][y, x] = value
    sw = P.SoftSweep(wl.rig, lv)
    r, c, aux = sw.forward(dev)
    one = torch.ones_like(r)
    pad = 16 * w
    buf = torch.zeros(2 * pad + h * w, device="cuda")
    g = [buf[pad:pad + h * w]] + [torch.zeros_like(d) for d in dev[1:]]
    gp = torch.zeros((2, 6), dtype=torch.float64, device="cuda")
    ims, poses = sw._args(dev, None)
    ptrs = (type(ims))(*[t.data_ptr() for t in g])
    assert P.load().psdiff_backward(sw.h, ims, poses, aux.data_ptr(), one.data_ptr(), one.data_ptr(), ptrs, gp.data_ptr(),
                                    torch.cuda.current_stream().cuda_stream) == P.PS_OK
    assert (buf[:pad] == 0).all() and (buf[pad + h * w:] == 0).all()
    bad = ~torch.isfinite(g[0].view(h, w))
    bad[y, x] = False
    assert not bad.any() and (g[0].nan_to_num(0, 0, 0) != 0).any()

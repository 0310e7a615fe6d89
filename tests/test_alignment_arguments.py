"""Grids that do not start where the kernels' vector accesses need them to are
refused before any CUDA call (and taken when they do: then the call goes on
to the first thing that only a well-formed pose passes)."""
import ctypes as C

import pytest

import paper_1809_06132_gb300 as P
from paper_1809_06132_gb300 import psweep as B

BUF = (C.c_double * 8192)()
BASE = (C.addressof(BUF) + 255) // 256 * 256


def _common(bad_pose):
    cam = B.ps_camera(xi=1.0, fx=8.0, fy=8.0, cx=4.0, cy=4.0, r2_max=1e30, width=8, height=8)
    pose = B.ps_pose()
    pose.R[0] = pose.R[4] = pose.R[8] = 1.0
    if bad_pose:
        pose.t[0] = float("nan")
    return (C.c_int32 * 3)(8, 8, 8), (C.c_double * 3)(), cam, pose


def _backward(grid, voxels, g_out, g_in, bad_pose=False):
    d, o, cam, pose = _common(bad_pose)
    f = P.load().tsdf_dense_fuse_backward_grid if grid else P.load().tsdf_dense_fuse_backward
    st = f(BASE + voxels, d, o, 0.1, 0.3, 4.0, BASE, C.byref(cam), C.byref(pose), BASE + g_out, BASE + g_in, BASE, BASE, None)
    return st, P.load().ps_last_error()


@pytest.mark.parametrize("grid,voxels,g_out,g_in", [(True, 4, 0, 0), (True, 0, 4, 0), (True, 0, 0, 4), (True, 0, 8, 2),
                                                    (False, 4, 0, 0)])
def test_backward_refuses_pairs_off_8_bytes(grid, voxels, g_out, g_in):
    st, msg = _backward(grid, voxels, g_out, g_in)
    assert st == P.PS_ERR_ARG and b"align" in msg


@pytest.mark.parametrize("grid,voxels,g_out,g_in", [(True, 8, 8, 24), (False, 8, 4, 4)])
def test_backward_takes_aligned_pointers(grid, voxels, g_out, g_in):
    st, msg = _backward(grid, voxels, g_out, g_in, bad_pose=True)
    assert st == P.PS_ERR_ARG and b"pose" in msg


@pytest.mark.parametrize("offset", [4, 8, 12])
def test_forward_refuses_grids_off_16_bytes(offset):
    d, o, cam, pose = _common(False)
    L = P.load()
    assert L.tsdf_integrate_dense_static(BASE + offset, d, o, 0.1, 0.3, 4.0, BASE, C.byref(cam), C.byref(pose),
                                         None) == P.PS_ERR_ARG
    assert b"align" in L.ps_last_error()

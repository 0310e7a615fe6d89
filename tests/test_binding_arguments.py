"""What the Python binding accepts and refuses before any library call."""
from types import SimpleNamespace as NS

import numpy as np
import pytest

from paper_1809_06132_gb300 import psweep as B


@pytest.mark.parametrize("R,t", [([2.0], np.zeros(3)), (2.0, np.zeros(3)), (np.eye(3), [0.5]), (np.eye(3), 0.5),
                                 (np.eye(3)[:2], np.zeros(3)), (np.eye(3), np.zeros(2)), ([], np.zeros(3))])
def test_a_pose_with_too_few_values_is_refused(R, t):
    with pytest.raises(IndexError):
        B.pose(NS(R=R, t=t))


@pytest.mark.parametrize("R,t", [(np.arange(9.0).reshape(3, 3), np.arange(3.0)), (list(range(9)), (0, 1, 2)),
                                 (np.arange(9.0, dtype=np.float32).reshape(3, 3).T.copy().T, [[0.0], [1.0], [2.0]]),
                                 (np.arange(9.0), [0.0, 1.0, 2.0, 1.0])])
def test_a_pose_keeps_its_values(R, t):
    p = B.pose(NS(R=R, t=t))
    assert list(p.R) == list(range(9)) and list(p.t) == [0.0, 1.0, 2.0]


@pytest.mark.parametrize("boxes,rows", [
    (None, []), (np.zeros((0, 4)), []), ([], []), ([(1, 2, 3, 4)], [(1, 2, 3, 4)]),
    (np.array([[1, 2, 3, 4], [5, 6, 7, 8]], dtype=np.int64), [(1, 2, 3, 4), (5, 6, 7, 8)]),
    (np.arange(8).reshape(4, 2).T, [(0, 2, 4, 6), (1, 3, 5, 7)]),
    ([(1, 2, 3)], [(1, 2, 3, 0)]), (np.array([[7], [8]]), [(7, 0, 0, 0), (8, 0, 0, 0)])])
def test_boxes_keep_their_values(boxes, rows):
    arr, n = B.boxes_array(boxes)
    assert n == len(rows) and len(arr) == max(1, n)
    assert [(b.x0, b.y0, b.x1, b.y1) for b in arr[:n]] == rows


@pytest.mark.parametrize("boxes", [[1, 2, 3, 4], [(1, 2, 3, 4, 5)], np.ones((1, 2, 2), dtype=np.int32)])
def test_other_shapes_of_boxes_are_refused(boxes):
    with pytest.raises(TypeError):
        B.boxes_array(boxes)

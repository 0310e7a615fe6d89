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

"""The benchmark's ground truth is checked against a scan that shares no screen with it."""
import os
import sys

import numpy as np
import pytest

torch = pytest.importorskip("torch")
sys.path.insert(0, os.path.dirname(os.path.dirname(os.path.abspath(__file__))))
import bench  # noqa: E402


class FakeIndex:
    """bruteforce and the plain scan of all cones; `wrong`: a query that linear search answers
    otherwise."""
    NC = 480

    def __init__(self, wrong=None):
        self.wrong = wrong

    def bruteforce(self, q, k):
        ids = q[:, :k].round().long()
        if self.wrong is not None:
            ids[self.wrong] += 1
        return ids, q[:, :k].clone()

    def search(self, q, P, k, path):
        assert P == self.NC and path == "plain"
        return q[:, :k].round().long(), q[:, :k].clone()


def test_linear_truth():
    q = torch.arange(0.0, 6000.0).reshape(1000, 6)
    ids, d2 = bench.linear_truth(FakeIndex(), q, 3)
    assert ids.shape == d2.shape == (1000, 3) and np.array_equal(ids, d2.astype(np.int64))
    with pytest.raises(RuntimeError):
        bench.linear_truth(FakeIndex(wrong=0), q, 3)
    with pytest.raises(RuntimeError):
        bench.linear_truth(FakeIndex(wrong=slice(480, 600)), q, 1)
    assert bench.linear_truth(FakeIndex(), q[:5], 2)[0].shape == (5, 2)

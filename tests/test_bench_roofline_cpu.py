"""The arithmetic that bench.py's roofline counts: every triple product once, however often its value is stored."""
import os
import sys

import numpy as np
import pytest

from . import _cases as CS

sys.path.insert(0, os.path.dirname(os.path.dirname(os.path.abspath(__file__))))


@pytest.mark.parametrize("N,R", [(64, 1), (64, 8), (64, 18), (128, 9), (128, 16)])
def test_distinct_products(N, R):
    """The distinct (w, {u, v}) among the used pairs whose second offset is an offset too; all others as they are."""
    import bench
    wv = CS.used_pairs(N, R).astype(np.int64)
    u = wv[:, :2] - wv[:, 2:]
    both = (u * u).sum(1) <= R * R
    lo = np.where(((u[:, 1] < wv[:, 3]) | ((u[:, 1] == wv[:, 3]) & (u[:, 0] < wv[:, 2])))[:, None], u, wv[:, 2:])
    want = (~both).sum() + len({tuple(r) for r in np.hstack([wv[both, :2], lo[both]])})
    r = CS.FC * N
    assert bench.distinct_products(int(r), r * r, R) == want

"""The mixed force kernel's variant 0 with long shares, straight and through the TMA ring: the
same FP32 sums, so they agree to the two-sum additions that join them
(tests/test_gpu_force_columns.py)."""
import numpy as np
import pytest

import ics
from tests.nbtools import condition_scales
from tests.test_gpu_force_columns import JOIN, _forces, _near, nb  # noqa: F401

pytestmark = pytest.mark.gpu


def test_straight_and_through_the_ring(nb):  # noqa: F811
    """Variants 0 and 5 form the same FP32 sums; variant 0 takes the ring itself for long ranges."""
    for n, splits in ((9001, (1, 2, 3)), (40000, (1, 5, 40)), (600001, (1, 20, 200))):
        snap = ics.plummer(n, seed=n, eps=1.0 / 64)
        idx = np.array([0, 1, n // 2, n - 2, n - 1], dtype=np.int32)
        A, K = condition_scales(snap.m, snap.x, snap.v, snap.eps2, idx)
        with nb.Context() as c:
            c.init(snap)
            for split in splits:
                a, b = _forces(nb, c, 0, split, idx), _forces(nb, c, 5, split, idx)
                for x, y, scale in zip(a, b, (A, K, np.abs(b[2]))):
                    _near(x, y, scale, JOIN, (n, split))

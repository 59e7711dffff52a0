"""The mixed force kernel's variant 0 with long shares, straight and through the TMA ring: the
same FP32 sums, so they agree to the two-sum additions that join them
(tests/test_gpu_force_columns.py); and the last sums of a few partials, against the FP64
oracle with the mixed path's tolerance."""
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


def test_few_partials(nb, orc):  # noqa: F811
    """The last sums of two, three, four and five partials, for one, two and eight particles."""
    n = 5000
    snap = ics.plummer(n, seed=8, eps=1.0 / 64)
    idx = np.linspace(0, n - 1, 23).astype(np.int32)
    ref = orc.force(snap.m, snap.x, snap.v, snap.eps2, idx)
    A, K = condition_scales(snap.m, snap.x, snap.v, snap.eps2, idx)
    with nb.Context() as c:
        c.init(snap)
        for variant in (0, 1, 2):
            for split in (1, 2, 3, 4, 5):
                for s in (1, 2, 8, 9, 23):
                    got = _forces(nb, c, variant, split, idx[:s])
                    for x, y, scale in zip(got, ref, (A, K, np.abs(ref[2]))):
                        _near(x, y[:s], scale[:s], 1e-6, (variant, split, s))

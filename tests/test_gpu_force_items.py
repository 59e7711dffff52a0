"""The mixed force kernel's whole items (variants 1 and 2) at the lengths where they meet the
columns: shares around 32, 64 and 128 tiles, odd block sizes, and blocks on both sides of the
line between the two; variant 0 with long shares, straight and through the TMA ring. Against
the FP64 oracle with the mixed path's tolerance, and against the same particles in a block
that goes to the other form: the FP32 sums are the same, so they agree to the two-sum
additions that join them (tests/test_gpu_force_columns.py)."""
import numpy as np
import pytest

import ics
from tests.nbtools import condition_scales
from tests.test_gpu_force_columns import JOIN, _forces, _near, nb  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("tiles", [33, 63, 64, 65, 66, 97, 127, 128, 129])
def test_items_and_columns(nb, orc, tiles):  # noqa: F811
    n = 256 * tiles - 7
    snap = ics.plummer(n, seed=tiles, eps=1.0 / 64)
    pick = np.unique(np.concatenate([np.arange(n - 20, n), np.linspace(0, n - 21, 500).astype(int)])).astype(np.int32)
    ar, kr, pr = orc.force(snap.m, snap.x, snap.v, snap.eps2, pick, nthreads=orc.default_threads())
    A, K = condition_scales(snap.m, snap.x, snap.v, snap.eps2, pick)
    with nb.Context() as c:
        c.init(snap)
        for variant in (1, 2):
            # many particles: items where a share has up to 128 tiles; few: columns above 32
            many = _forces(nb, c, variant, 1, pick)
            for got, ref, scale in zip(many, (ar, kr, pr), (A, K, np.abs(pr))):
                _near(got, ref, scale, 1e-6, (tiles, variant))
            for s in (1, 2, 7, 9, 40, 101, 255, 501):
                pos = np.linspace(0, len(pick) - 1, s).astype(int)
                few = _forces(nb, c, variant, 1, pick[pos])
                for got, ref, scale in zip(few, many, (A, K, np.abs(pr))):
                    _near(got, ref[pos], scale[pos], JOIN, (tiles, variant, s))
            two = _forces(nb, c, variant, 2, pick[:201])     # shares of half the length
            for got, ref, scale in zip(two, (ar, kr, pr), (A, K, np.abs(pr))):
                _near(got, ref[:201], scale[:201], 1e-6, (tiles, variant, "split"))


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

"""The mixed force kernel's columns (variants 1 to 4): blocks, splits and particle counts
at the edges of its units (odd and short shares, a half-filled last row, several units
side by side, runs over several i-blocks, ranges of j), against the FP64 oracle with the
mixed path's tolerances (tests/test_gpu_parity.py), and against themselves: which FP32
sums are formed depends on the variant and the split only, not on the block, so a
particle's sums in blocks of different sizes agree to the two-sum additions that join
them: below 600 additions with an error of 2^-46 of a partial each, 1e-11 of the
condition scale."""
import numpy as np
import pytest

import ics
from tests.nbtools import condition_scales

pytestmark = pytest.mark.gpu

JOIN = 1e-11


@pytest.fixture(scope="module")
def nb():
    import paper_0711_0643_gb300 as pkg
    pkg.build()
    from paper_0711_0643_gb300 import nbody
    nbody.load()
    return nbody


def _forces(nb, c, variant, split, idx, rng=None):
    for b in range(32):
        nb.nb_set_tuning(c.ctx, b, variant, split)
    if rng is None:
        return nb.nb_force_jerk(c.ctx, idx)
    return nb.nb_force_jerk_range(c.ctx, idx, len(idx), *rng)


def _near(x, y, scale, tol, where):
    d = np.abs(x - y).reshape(len(scale), -1).max(axis=1)
    assert np.all(d <= tol * scale), (where, (d / scale).max())


@pytest.mark.parametrize("n", [1500, 5000, 16384, 33000, 70001])
def test_columns(nb, orc, n):
    snap = ics.plummer(n, seed=n, eps=1.0 / 64)
    pick = np.unique(np.concatenate([np.arange(n - 40, n), np.linspace(0, n - 41, 560).astype(int)])).astype(np.int32)
    ar, kr, pr = orc.force(snap.m, snap.x, snap.v, snap.eps2, pick, nthreads=orc.default_threads())
    A, K = condition_scales(snap.m, snap.x, snap.v, snap.eps2, pick)
    with nb.Context() as c:
        c.init(snap)
        for variant in (1, 2, 3, 4):
            for split in (1, 3, 16, 50):
                a, k, phi = _forces(nb, c, variant, split, pick)
                _near(a, ar, A, 1e-6, (n, variant, split, "a"))
                _near(k, kr, K, 1e-6, (n, variant, split, "k"))
                _near(phi, pr, np.abs(pr), 1e-6, (n, variant, split, "phi"))
                # the split is kept per bucket in proportion to the block: the same one for
                # every size is asked for by a bucket of its own
                for s in (1, 2, 7, 8, 9, 31, 33, 64, 65, 130, 257):
                    I = {1: 2, 2: 8, 3: 32, 4: 256}[variant]
                    top = 1 << (s - 1).bit_length()
                    if -(-min(top, n) // I) != -(-s // I):
                        continue   # the kernel would scale the split
                    pos = np.linspace(0, len(pick) - 1, s).astype(int)
                    b = _forces(nb, c, variant, split, pick[pos])
                    whole = -(-min(1 << (len(pick) - 1).bit_length(), n) // I) == -(-len(pick) // I)
                    if whole:
                        _near(b[0], a[pos], A[pos], JOIN, (n, variant, split, s, "a"))
                        _near(b[1], k[pos], K[pos], JOIN, (n, variant, split, s, "k"))
                        _near(b[2], phi[pos], np.abs(pr[pos]), JOIN, (n, variant, split, s, "phi"))
                    _near(b[0], ar[pos], A[pos], 1e-6, (n, variant, split, s, "a"))
                    _near(b[1], kr[pos], K[pos], 1e-6, (n, variant, split, s, "k"))


@pytest.mark.parametrize("variant", [0, 1, 2, 3, 4])
def test_ranges(nb, orc, variant):
    n = 20000
    snap = ics.plummer(n, seed=5, eps=1.0 / 64)
    with nb.Context() as c:
        c.init(snap)
        for s in (1, 10, 300):
            idx = np.unique(np.linspace(0, n - 1, s).astype(np.int32))
            ar, kr, pr = orc.force(snap.m, snap.x, snap.v, snap.eps2, idx, nthreads=orc.default_threads())
            A, K = condition_scales(snap.m, snap.x, snap.v, snap.eps2, idx)
            cuts = (0, 256, 3 * 256, 40 * 256, n)
            parts = [_forces(nb, c, variant, 3, idx, r) for r in zip(cuts, cuts[1:])]
            _near(sum(p[0] for p in parts), ar, A, 1e-6, (variant, s))
            _near(sum(p[1] for p in parts), kr, K, 1e-6, (variant, s))
            again = [_forces(nb, c, variant, 3, idx, r) for r in zip(cuts, cuts[1:])]
            for p, q in zip(parts, again):
                assert all(np.array_equal(x, y) for x, y in zip(p, q))   # the same bits again


def test_every_particle(nb, orc):
    """s = N: runs of many i-blocks, whole i-blocks in one CTA, every self pair."""
    for n in (700, 9001):
        snap = ics.plummer(n, seed=n, eps=0.0)
        idx = np.arange(n, dtype=np.int32)
        with nb.Context() as c:
            c.init(snap)
            ref = orc.force(snap.m, snap.x, snap.v, 0.0, idx, nthreads=orc.default_threads())
            A, K = condition_scales(snap.m, snap.x, snap.v, 0.0, idx)
            for variant in (1, 2, 3, 4):
                a, k, phi = _forces(nb, c, variant, 1, idx)
                _near(a, ref[0], A, 1e-6, (n, variant))
                _near(k, ref[1], K, 1e-6, (n, variant))

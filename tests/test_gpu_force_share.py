"""The mixed force kernel with its records resident in shared memory (variant 6, clusters
of eight CTAs): particle counts at the edges of the 256-record copies and of the padding to
32 records (CTAs without a record among them), blocks at the edges of the passes and of the
256-position chunks (one, several and many chunks per cluster), and ranges of j. Against the
FP64 oracle with the mixed path's tolerances (tests/test_gpu_parity.py), and bit for bit
against a second call."""
import numpy as np
import pytest

import ics
from tests.nbtools import condition_scales

pytestmark = pytest.mark.gpu

PASSES = (1, 2, 3, 4, 5, 8, 9, 16, 31, 33, 64, 129, 255)


@pytest.fixture(scope="module")
def nb():
    import paper_0711_0643_gb300 as pkg
    pkg.build()
    from paper_0711_0643_gb300 import nbody
    nbody.load()
    return nbody


def _check(nb, c, snap, idx, ref, scales, where, rng=None):
    def call():
        if rng is None:
            return nb.nb_force_jerk(c.ctx, idx)
        out = [nb.nb_force_jerk_range(c.ctx, idx, len(idx), *r) for r in rng]
        return tuple(sum(o[q] for o in out) for q in range(3))
    got, again = call(), call()
    for g, b in zip(got, again):
        np.testing.assert_array_equal(g, b)
    for g, r, sc, name in zip(got, ref, scales, "akp"):
        d = np.abs(g - r).reshape(len(idx), -1).max(axis=1)
        assert np.all(d <= 1e-6 * sc), (where, name, (d / sc).max())


@pytest.mark.parametrize("n", [2, 65, 511, 4095, 4098, 8191, 12300, 16384])
def test_share(nb, orc, n):
    snap = ics.plummer(n, seed=n, eps=1.0 / 64)
    allidx = np.arange(n, dtype=np.int32)
    pick = np.linspace(0, n - 1, min(n, 600)).astype(np.int32)
    ar, kr, pr = orc.force(snap.m, snap.x, snap.v, snap.eps2, pick, nthreads=orc.default_threads())
    A, K = condition_scales(snap.m, snap.x, snap.v, snap.eps2, pick)
    P = np.abs(pr)
    with nb.Context() as c:
        c.init(snap)
        for b in range(32):
            nb.nb_set_tuning(c.ctx, b, 6, 1)
        # per cluster 1, 2, ... positions, whatever the number of clusters: blocks from one
        # particle to all of them
        for s in PASSES + (300, 600):
            q = np.unique(np.linspace(0, len(pick) - 1, min(s, len(pick))).astype(int))
            _check(nb, c, snap, pick[q], (ar[q], kr[q], pr[q]), (A[q], K[q], P[q]), (n, s))
        # blocks of several passes and chunks per cluster
        for m in (PASSES[-1] * 18 + 7, 256 * 40 + 11):
            m = min(m, n)
            if m <= len(pick):
                continue
            idx = np.unique(np.concatenate([pick, allidx[:m]])).astype(np.int32)
            a, k, p = nb.nb_force_jerk(c.ctx, idx)
            for x, y in zip((a, k, p), nb.nb_force_jerk(c.ctx, idx)):
                np.testing.assert_array_equal(x, y)
            pos = np.searchsorted(idx, pick)
            for g, r, sc, name in ((a, ar, A, "a"), (k, kr, K, "k"), (p, pr, P, "p")):
                d = np.abs(g[pos] - r).reshape(len(pick), -1).max(axis=1)
                assert np.all(d <= 1e-6 * sc), (n, m, name, (d / sc).max())


def test_share_ranges(nb, orc):
    n = 40000   # too many records for the shares as a whole, each range fits
    snap = ics.plummer(n, seed=8, eps=1.0 / 64)
    with nb.Context() as c:
        c.init(snap)
        for b in range(32):
            nb.nb_set_tuning(c.ctx, b, 6, 1)
        for s in (1, 3, 40, 700):
            idx = np.unique(np.linspace(0, n - 1, s).astype(np.int32))
            ar, kr, pr = orc.force(snap.m, snap.x, snap.v, snap.eps2, idx, nthreads=orc.default_threads())
            A, K = condition_scales(snap.m, snap.x, snap.v, snap.eps2, idx)
            cuts = (0, 256, 512 + 256 * 15, 20480, 36864, n)
            _check(nb, c, snap, idx, (ar, kr, pr), (A, K, np.abs(pr)), s, list(zip(cuts, cuts[1:])))

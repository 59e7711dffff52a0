"""The FP64 force kernel's equal runs of (i-block, j unit) pairs: block sizes and
particle counts at the edges of its i-blocks and units, with one and many CTAs to an
i-block, over ranges of j, and pair distances outside the FP32 exponent range.
Tolerance: the FP64 path's 1e-12 relative (tests/test_gpu_parity.py)."""
import numpy as np
import pytest

import ics
from tests.nbtools import condition_scales, rel_errors, rel_scalar

pytestmark = pytest.mark.gpu

TOL = 1e-12


@pytest.fixture(scope="module")
def nb():
    import paper_0711_0643_gb300 as pkg
    pkg.build()
    from paper_0711_0643_gb300 import nbody
    nbody.load()
    return nbody


def _check(snap, idx, got, ref, where):
    A, K = condition_scales(snap.m, snap.x, snap.v, snap.eps2, idx)
    ea, ek = rel_errors(got[0], ref[0], A), rel_errors(got[1], ref[1], K)
    ep = rel_scalar(got[2], ref[2])
    assert ea.max() < TOL and ek.max() < TOL and ep.max() < TOL, (where, ea.max(), ek.max(), ep.max())


def _pick(n, s):
    return np.unique(np.linspace(0, n - 1, s).astype(np.int32))


@pytest.mark.parametrize("n", [1, 31, 255, 257, 1000, 4099])
def test_block_edges(nb, orc, n):
    snap = ics.random_state(n, seed=n, eps=0.01)
    with nb.Context(precision=nb.NB_PREC_FP64) as c:
        c.init(snap)
        for s in sorted({min(s, n) for s in (1, 2, 3, 15, 16, 17, 31, 32, 33, 64, 65, 255, 256, 257, 1023, n)}):
            idx = _pick(n, s)
            ref = orc.force(snap.m, snap.x, snap.v, snap.eps2, idx)
            for variant, split in ((-1, 1), (0, 1), (0, 64), (1, 1), (1, 7), (1, 100000)):
                for b in range(32):
                    nb.nb_set_tuning(c.ctx, b, variant, split)
                _check(snap, idx, nb.nb_force_jerk(c.ctx, idx), ref, (n, s, variant, split))


def test_ranges_add_up(nb, orc):
    n = 2000
    snap = ics.plummer(n, seed=3, eps=1.0 / 64)
    with nb.Context(precision=nb.NB_PREC_FP64) as c:
        c.init(snap)
        for s in (1, 40, 700):
            idx = _pick(n, s)
            ref = orc.force(snap.m, snap.x, snap.v, snap.eps2, idx)
            cuts = (0, 256, 1536, 1792, n)
            parts = [nb.nb_force_jerk_range(c.ctx, idx, s, lo, hi) for lo, hi in zip(cuts, cuts[1:])]
            _check(snap, idx, [sum(p[q] for p in parts) for q in range(3)], ref, s)
            again = nb.nb_force_jerk(c.ctx, idx)
            for x, y in zip(again, nb.nb_force_jerk(c.ctx, idx)):
                assert np.array_equal(x, y)


@pytest.mark.parametrize("scale", [2.0 ** -80, 2.0 ** -61, 2.0 ** -58, 2.0 ** 58, 2.0 ** 61, 2.0 ** 80])
def test_distances_outside_fp32(nb, orc, scale):
    snap = ics.random_state(300, seed=9, eps=0.0)
    snap.x *= scale
    with nb.Context(precision=nb.NB_PREC_FP64, dt_min=2.0 ** -300, dt_max=2.0 ** 300) as c:
        c.init(snap)
        idx = _pick(300, 50)
        _check(snap, idx, nb.nb_force_jerk(c.ctx, idx), orc.force(snap.m, snap.x, snap.v, 0.0, idx), scale)

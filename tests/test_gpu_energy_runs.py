"""The energy kernel's equal runs of (i-block, j unit) pairs at the edges of its blocks
(128 particles) and units (32), every pair counted once, against the FP64 oracle.
Tolerance: a pair term is within 2^-43 and the FP64 sums within 1e-15 relative of the
(one-signed) sum: 1e-12 holds with a wide margin; K is FP64 throughout (1e-14)."""
import numpy as np
import pytest

import ics

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def nb():
    import paper_0711_0643_gb300 as pkg
    pkg.build()
    from paper_0711_0643_gb300 import nbody
    nbody.load()
    return nbody


@pytest.mark.parametrize("n", [1, 2, 3, 31, 32, 33, 64, 127, 128, 129, 160, 161, 255, 256, 257, 385, 1000, 2049, 5000])
@pytest.mark.parametrize("eps", [0.0, 1.0 / 64])
def test_energy_edges(nb, orc, n, eps):
    snap = ics.random_state(n, seed=50 + n, eps=eps)
    snap.x[:, 0] += 3.0            # off-centre: the low halves of the positions matter
    for prec in (nb.NB_PREC_MIXED, nb.NB_PREC_FP64):
        with nb.Context(precision=prec) as c:
            c.init(snap)
            E, K, W = nb.nb_energy(c.ctx)
            Kr, Wr = orc.energy(snap.m, snap.x, snap.v, snap.eps2)
            assert abs(K - Kr) <= 1e-14 * abs(Kr)
            assert abs(W - Wr) <= 1e-12 * abs(Wr)
            assert E == K + W
            assert nb.nb_energy(c.ctx) == (E, K, W)   # the same bits again


def test_close_pair_far_from_the_origin(nb, orc):
    """Two particles 1e-6 apart at |x| = 1 among others: the pair's distance lives in the low halves."""
    snap = ics.random_state(200, seed=4, eps=0.0)
    snap.x[7] = np.array([1.0, -1.0, 0.5])
    snap.x[150] = snap.x[7] + np.array([1e-6, 0.0, 0.0])
    with nb.Context() as c:
        c.init(snap)
        W = nb.nb_energy(c.ctx)[2]
    # the positions' double-single copies are within 2^-49 of each coordinate: 2^-48 / 1e-6 of this pair's distance
    assert abs(W - orc.energy(snap.m, snap.x, snap.v, 0.0)[1]) <= 8e-9 * abs(W)

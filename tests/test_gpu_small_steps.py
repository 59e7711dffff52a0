"""Small blocks in the engine and the ensemble: systems without softening (the self pair
must be left out by index there, and only there), with a softening too small for the
self pair's terms to be finite, and the ensemble's buffers taken over by the next
ensemble of the context. Energy tolerances as in tests/test_gpu_ensemble.py: twice the
oracle's error plus 1e-9; taken-over buffers give the bits of fresh ones."""
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


def _pack(members):
    off = np.zeros(len(members) + 1, dtype=np.int64)
    off[1:] = np.cumsum([s.n for s in members])
    return (off, np.concatenate([s.m for s in members]), np.concatenate([s.x for s in members]),
            np.concatenate([s.v for s in members]), np.array([s.eps2 for s in members]))


def _oracle_error(orc, s, t_end):
    o = orc.System(s.m, s.x, s.v, s.eps2, nthreads=orc.default_threads())
    e0 = o.energy()
    assert o.run(t_end) == 0
    return abs(o.energy() - e0) / abs(e0)


@pytest.mark.parametrize("eps", [0.0, 1e-25, 1e-15, 1.0 / 64])
def test_engine_softenings(nb, orc, eps):
    for n in (5, 150, 1100):
        s = ics.plummer(n, seed=60 + n, eps=eps)
        with nb.Context() as c:
            c.init(s)
            assert nb.nb_get_engine(c.ctx)[0] > 0
            e0 = nb.nb_energy(c.ctx)[0]
            nb.nb_run(c.ctx, 1.0 / 16)
            st = c.state()
            assert all(np.all(np.isfinite(st[k])) for k in ("x", "v", "a", "k", "dt"))
            assert abs(nb.nb_energy(c.ctx)[0] - e0) / abs(e0) <= 2 * _oracle_error(orc, s, 1.0 / 16) + 1e-9


@pytest.mark.parametrize("eps", [0.0, 1e-25, 1.0 / 64])
def test_ensemble_softenings(nb, orc, eps):
    mem = [ics.plummer(n, seed=80 + n, eps=eps) for n in (2, 30, 200, 700)]
    off, m, x, v, e2 = _pack(mem)
    with nb.Context() as c:
        nb.nb_ensemble_init(c.ctx, off, m, x, v, e2)
        e0 = nb.nb_ensemble_energy(c.ctx, len(mem))
        nb.nb_ensemble_run(c.ctx, 1.0 / 16)
        e1 = nb.nb_ensemble_energy(c.ctx, len(mem))
    for q, s in enumerate(mem):
        assert abs(e1[q] - e0[q]) / abs(e0[q]) <= 2 * _oracle_error(orc, s, 1.0 / 16) + 1e-9, (q, s.n)


def test_ensemble_buffers_taken_over(nb):
    sizes = [(300, 900, 40), (250, 800), (300, 900, 40), (10, 20), (500, 600, 700, 800), (64,), (64,)]
    kept = nb.Context()
    for q, ns in enumerate(sizes):
        mem = [ics.plummer(n, seed=7 * n + q, eps=1.0 / 64) for n in ns]
        off, m, x, v, e2 = _pack(mem)
        got = []
        for c in (kept, nb.Context()):
            nb.nb_ensemble_init(c.ctx, off, m, x, v, e2)
            e0 = nb.nb_ensemble_energy(c.ctx, len(mem))
            nb.nb_ensemble_run(c.ctx, 1.0 / 16)
            got.append((e0, nb.nb_ensemble_energy(c.ctx, len(mem)), *nb.nb_ensemble_stats(c.ctx, len(mem)),
                        nb.nb_ensemble_get_shape(c.ctx), *nb.nb_ensemble_get_state(c.ctx, int(off[-1])).values()))
            if c is not kept:
                c.close()
        for a, b in zip(*got):
            assert np.array_equal(a, b), (q, ns)
    kept.close()

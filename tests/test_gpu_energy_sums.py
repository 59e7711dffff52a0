"""The energy's sums where their arithmetic could give out, against direct FP64 sums: odd
particle counts far from the origin (the last record of two particles is half empty, and
nothing in the other half may reach the sum), and rows of half a million terms that do not
average out over the particles."""
import math

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


@pytest.mark.parametrize("n", [1, 3, 33, 127, 129, 161, 1001])
def test_odd_count_far_from_the_origin(nb, orc, n):
    """Coordinates around 2^68 on a grid of 2^50 (exact as double-single), separations up to
    2^57: every pair's r^2 is an ordinary FP32 number, the squared distance to anything near
    the origin is not. Tolerance as in tests/test_gpu_energy_runs.py: 1e-12 (W), 1e-14 (K)."""
    rng = ics.SplitMix64(700 + n)
    cells = np.unique(rng.next_u64(4 * n) % (1 << 18))      # different places on a 64^3 grid
    cells = cells[np.argsort(rng.next_u64(len(cells)))][:n].astype(np.int64)
    x = np.stack([cells & 63, (cells >> 6) & 63, cells >> 12], axis=1) * 2.0 ** 50 + 2.0 ** 68 * np.array([1.0, -1.0, 0.5])
    v = rng.uniform(3 * n).reshape(n, 3) - 0.5
    m = (0.5 + rng.uniform(n)) / n
    Kr, Wr = orc.energy(m, x, v, 0.0)
    with nb.Context(precision=nb.NB_PREC_FP64) as c:
        nb.nb_init(c.ctx, m, x, v, 0.0)
        E, K, W = nb.nb_energy(c.ctx)
    assert abs(K - Kr) <= 1e-14 * abs(Kr)
    assert abs(W - Wr) <= 1e-12 * abs(Wr)      # n = 1: both are 0
    assert E == K + W


@pytest.mark.parametrize("seed", [1, 2, 3])
def test_one_heavy_body_holds_a_long_row(nb, seed):
    """Body 0 holds all but 2^-51 of the mass, so W is its own row to 2^-51. Tolerance: a pair
    term is within 2^-43, and the row's additions leave below 1e-13 (2^18 terms a lane, rms
    in an FP32 emulation): 1e-12."""
    n, eps = (1 << 19) + 3, 1.0 / 64
    rng = ics.SplitMix64(900 + seed)
    x = rng.uniform(3 * n).reshape(n, 3) * 2.0 - 1.0
    v = rng.uniform(3 * n).reshape(n, 3) - 0.5
    m = 2.0 ** -70 * (0.5 + rng.uniform(n))
    m[0] = 1.0
    r = np.sqrt(((x[1:] - x[0]) ** 2).sum(1) + eps * eps)
    Wr = -math.fsum(m[1:] / r)
    Kr = 0.5 * math.fsum(m * (v * v).sum(1))
    with nb.Context() as c:
        nb.nb_init(c.ctx, m, x, v, eps * eps)
        E, K, W = nb.nb_energy(c.ctx)
    assert abs(K - Kr) <= 1e-14 * Kr
    assert abs(W - Wr) <= 1e-12 * abs(Wr), (W - Wr) / Wr

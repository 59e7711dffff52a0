"""Perturber lists where the FP32 test cannot decide, and around it: stars at the
threshold distance to within 1e-2 ... 1e-15 (relative), systems far from the origin
(positions that need their low halves), positions and masses scaled out of the FP32
test's range, zero masses and coincident members, for one, two and four binaries to a
CTA. The lists and counts are whole numbers: equal to the FP64 oracle's."""
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


def _equal(nb, orc, m, x, pairs, gamma, nmax):
    with nb.Context(precision=nb.NB_PREC_FP64, dt_min=2.0 ** -300, dt_max=2.0 ** 300) as c:
        nb.nb_init(c.ctx, m, x, np.zeros_like(x), 1.0)
        gl, gc = nb.nb_perturbers(c.ctx, pairs, gamma=gamma, nmax=nmax)
    ol, oc = orc.perturbers(m, x, pairs, gamma=gamma, nmax=nmax)
    np.testing.assert_array_equal(gc, oc)
    np.testing.assert_array_equal(gl, ol)
    return gc


def _threshold_system(nbin, seed, n_near=6000):
    """nbin binaries in a unit sphere; stars at the threshold distance of one of them."""
    rng = ics.SplitMix64(seed)
    n = 2 * nbin + n_near
    m = np.full(n, 1.0 / n)
    x = np.empty((n, 3))
    cm = rng.uniform(3 * nbin).reshape(nbin, 3) * 2.0 - 1.0
    d = 1e-4 * 10.0 ** (2.0 * rng.uniform(nbin))
    u = rng.uniform(3 * nbin).reshape(nbin, 3) - 0.5
    u /= np.linalg.norm(u, axis=1)[:, None]
    x[:nbin] = cm + 0.5 * d[:, None] * u
    x[nbin:2 * nbin] = cm - 0.5 * d[:, None] * u
    pairs = np.stack([np.arange(nbin), nbin + np.arange(nbin)], axis=1).astype(np.int32)
    gamma = 1e-7
    of = (rng.uniform(n_near) * nbin).astype(int)
    rc = d[of] * (2.0 * (1.0 / n) / (gamma * (2.0 / n))) ** (1.0 / 3.0)
    off = 10.0 ** (-2.0 - 13.0 * rng.uniform(n_near)) * np.where(rng.uniform(n_near) < 0.5, -1.0, 1.0)
    w = rng.uniform(3 * n_near).reshape(n_near, 3) - 0.5
    w /= np.linalg.norm(w, axis=1)[:, None]
    x[2 * nbin:] = cm[of] + (rc * (1.0 + off))[:, None] * w
    return m, x, pairs, gamma


# one binary to a CTA, one, two, four, four
@pytest.mark.parametrize("nbin", [1, 100, 700, 1300, 2500])
def test_stars_at_the_threshold(nb, orc, nbin):
    m, x, pairs, gamma = _threshold_system(nbin, 11 + nbin)
    counts = _equal(nb, orc, m, x, pairs, gamma, 256)
    assert counts.max() > 0
    _equal(nb, orc, m, x, pairs, gamma, 4096)


@pytest.mark.parametrize("shift", [1e3, 1e6, 1e9])
def test_far_from_the_origin(nb, orc, shift):
    m, x, pairs, gamma = _threshold_system(50, 5)
    _equal(nb, orc, m, x + np.array([shift, -shift, 0.5 * shift]), pairs, gamma, 256)


@pytest.mark.parametrize("px,pm", [(2.0 ** 20, 1.0), (2.0 ** -20, 1.0), (2.0 ** 90, 1.0), (2.0 ** -130, 1.0), (1.0, 2.0 ** 70),
                                   (1.0, 2.0 ** -70), (1.0, 2.0 ** -140), (2.0 ** -60, 2.0 ** -100)])
def test_scaled(nb, orc, px, pm):
    m, x, pairs, gamma = _threshold_system(20, 6, 1500)
    _equal(nb, orc, m * pm, x * px, pairs, gamma, 256)


def test_odd_members_and_masses(nb, orc):
    m, x, pairs, gamma = _threshold_system(8, 7, 700)
    m[20:200:7] = 0.0
    m[21:200:7] *= 1e-30
    m[22:200:7] *= 1e20
    x[300:310] = x[pairs[0, 0]]             # stars on a member
    x[pairs[1, 1]] = x[pairs[1, 0]]         # coincident members: no separation
    pairs[2] = pairs[2][::-1]
    pairs[3] = [707, 5]
    for gamma in (1e-7, 1e-3, 1e-12):
        _equal(nb, orc, m, x, pairs, gamma, 100)

"""Perturber lists in other units of mass: the FP32 test scales the masses by a power of two
where the first and the last star are both outside its range. Lists and counts equal to the
FP64 oracle's with stars at the threshold, on both sides of each limit of the scaling (2^-34
and 2^8, 2^-120 and 2^120), with the scale taken from a star that is not like the others,
and over a j-range; and the numbers of binaries at which a CTA takes more of them."""
import numpy as np
import pytest

from tests.test_gpu_perturbers_window import _equal, _threshold_system, nb  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("k", [-131, -120, -105, -40, -22, -21, -20, 19, 20, 21, 40, 101, 131, 134, 300])
def test_units_of_mass(nb, orc, k):  # noqa: F811
    """m = 2^k / n with n = 1540, so a star has the exponent k - 11."""
    m, x, pairs, gamma = _threshold_system(20, 40 + k, 1500)
    _equal(nb, orc, m * 2.0 ** k, x, pairs, gamma, 256)


@pytest.mark.parametrize("first,last", [(0.0, 2.0 ** 50), (2.0 ** 50, 0.0), (2.0 ** 90, 2.0 ** 60), (1.0, 2.0 ** 60), (2.0 ** 60, 1.0),
                                        (2.0 ** 20, 2.0 ** 200), (-(2.0 ** 60), 2.0 ** 40)])
def test_ends_unlike_the_rest(nb, orc, first, last):  # noqa: F811
    """The first and the last star (a member of no other binary than the first's) set the scale."""
    m, x, pairs, gamma = _threshold_system(9, 71, 900)
    m = m * 2.0 ** 60
    m[0], m[-1] = first, last
    _equal(nb, orc, m, x, pairs, gamma, 300)


def test_range(nb, orc):  # noqa: F811
    m, x, pairs, gamma = _threshold_system(30, 72, 2000)
    m = m * 2.0 ** 45
    m[100], m[899] = 1.0, 0.5
    with nb.Context(precision=nb.NB_PREC_FP64, dt_min=2.0 ** -300, dt_max=2.0 ** 300) as c:
        nb.nb_init(c.ctx, m, x, np.zeros_like(x), 1.0)
        for lo, hi in ((0, 100), (100, 900), (101, 899), (900, 2060), (500, 500)):
            gl, gc = nb.nb_perturbers(c.ctx, pairs, gamma=gamma, nmax=100, j_lo=lo, j_hi=hi)
            ol, oc = orc.perturbers(m, x, pairs, gamma=gamma, nmax=100, j_lo=lo, j_hi=hi)
            np.testing.assert_array_equal(gc, oc)
            np.testing.assert_array_equal(gl, ol)


@pytest.mark.parametrize("nbin", [607, 608, 609, 1215, 1216, 1217])
def test_binaries_per_cta(nb, orc, nbin):  # noqa: F811
    """One, two and four binaries to a CTA, the last CTA full and partly filled."""
    m, x, pairs, gamma = _threshold_system(nbin, 80 + nbin, 3000)
    _equal(nb, orc, m, x, pairs, gamma, 256)

"""Lattice totals from float sums with carried errors (lb_reduce): odd and
tiny lattices (paired loads and their tail), wide ranges of exponents, and
sums that leave the float range, against exactly rounded sums of the stored
values.

Bound: a thread's sum is exact to about 70 bits; the FP64 additions after it
(at most 19 rows, 5 + 5 levels of warp and block sums, 304 partials) round
fewer than 400 times, each by 2^-53 of a sum of magnitudes.
"""
import math

import numpy as np
import pytest

import lb_inputs as L
from tests.parity import P0

pytestmark = pytest.mark.gpu

BOUND = 400 * 2.0 ** -53


@pytest.fixture(scope="module", autouse=True)
def _setup():
    import paper_1405_6162_gb300 as lbpkg
    lbpkg.build()


def _check(lat, out):
    from paper_1405_6162_gb300 import VELOCITIES
    f, g = lat.get_state()
    c = VELOCITIES.astype(float)
    want = [math.fsum(f.ravel())] + [math.fsum((c[:, a, None] * f).ravel()) for a in range(3)] + [math.fsum(g.ravel())]
    size = [np.abs(f).sum()] * 4 + [np.abs(g).sum()]
    for k in range(5):
        assert abs(out[k] - want[k]) <= BOUND * size[k], (k, out[k], want[k])


@pytest.mark.parametrize("precision", ["fp32_shifted", "fp64_df", "fp64"])
@pytest.mark.parametrize("dims", [(1, 1, 1), (1, 1, 2), (3, 1, 1), (5, 7, 9), (64, 61, 59), (33, 97, 101)])
def test_totals(dims, precision):
    from paper_1405_6162_gb300 import Lattice
    n = int(np.prod(dims))
    w = np.array([1 / 3] + [1 / 18] * 6 + [1 / 36] * 12)[:, None]
    with Lattice.from_params(dims, P0, precision=precision) as lat:
        f = w + L.uniform(900, 19 * n, -0.02, 0.02).reshape(19, n) * 10.0 ** L.uniform(901, 19 * n, -12, 0).reshape(19, n)
        g = L.uniform(902, 19 * n, -1, 1).reshape(19, n) * 10.0 ** L.uniform(903, 19 * n, -20, 0).reshape(19, n)
        lat.set_state(f, g)
        _check(lat, lat.reduce())


@pytest.mark.parametrize("precision", ["fp32_shifted", "fp64_df"])
def test_sums_beyond_the_float_range(precision):
    from paper_1405_6162_gb300 import Lattice
    dims = (70, 60, 41)
    n = int(np.prod(dims))
    with Lattice.from_params(dims, P0, precision=precision) as lat:
        f = L.uniform(910, 19 * n, -1e38, 3e38).reshape(19, n)
        g = L.uniform(911, 19 * n, -3e38, 3e38).reshape(19, n)
        lat.set_state(f, g)
        _check(lat, lat.reduce())

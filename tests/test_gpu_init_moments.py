"""Start and read-out of float storage: the start's equilibria are the FP64
ones rounded once, whatever the size of phi0, and the moments divide by rho on
both sides of the range in which a float reciprocal starts the division."""
import numpy as np
import pytest

import lb_inputs as L
from tests.parity import P0

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _setup():
    import paper_1405_6162_gb300 as lbpkg
    lbpkg.build()


def _init(dims, precision, points, phi0, u0, **kw):
    from paper_1405_6162_gb300 import Lattice
    with Lattice.from_params(dims, dict(P0, **kw), precision=precision) as lat:
        lat.set_stencil(points)
        lat.init(phi0, u0)
        return lat.get_state()


# zeros of both signs, values whose split parts are normal floats, and values
# on either side of that range (2^-63), down to below the float range
VALUES = [0.0, -0.0, 0.3, -1.0, 1e-8, -2.0 ** -63, 1.1e-19, 1e-30, -1e-50, 0.01, 2.0 ** -62, -7.3e-5]


@pytest.mark.parametrize("points", [7, 19, 27])
@pytest.mark.parametrize("dims,flow", [((1, 1, 1), True), ((5, 3, 2), False), ((33, 7, 4), True)])
def test_float_start_is_the_fp64_equilibrium_rounded_once(dims, flow, points):
    n = dims[0] * dims[1] * dims[2]
    phi0 = np.resize(np.array(VALUES), n) * (1.0 + 1e-3 * L.uniform(300, n, -1, 1))
    u0 = 0.02 * L.uniform(301, 3 * n, -1, 1).reshape(3, n) if flow else None
    if flow:
        u0[0, ::2] = 0.0
    f64, g64 = _init(dims, "fp64", points, phi0, u0)
    f32, g32 = _init(dims, "fp32_shifted", points, phi0, u0)
    w = np.array([1 / 3] + [1 / 18] * 6 + [1 / 36] * 12)[:, None] * P0["rho0"]
    # half an ulp of the float, and the ~2^-46 of the double-float sums behind
    # it, whose terms are at most 1 (get_state adds w rho0 in FP64)
    assert (np.abs(g32 - g64) <= 2.0 ** -24 * np.abs(g64) + 2.0 ** -44).all()
    assert (np.abs(f32 - f64) <= 2.0 ** -24 * np.abs(f64 - w) + 2.0 ** -44).all()


@pytest.mark.parametrize("precision,tol", [("fp32_shifted", 1e-5), ("fp64_df", 1e-12)])
@pytest.mark.parametrize("rho0", [1.0, 1e-20, 1e31])
def test_velocity_of_small_and_large_densities(rho0, precision, tol):
    """1e31 > 2^100: divided in FP64.  Float sums of 19 values w (rho + ..):
    errors of a few 2^-24 of rho |u|, tol times the largest |u| = 0.02."""
    from paper_1405_6162_gb300 import Lattice
    dims, n = (9, 5, 4), 180
    u0 = 0.02 * L.uniform(302, 3 * n, -1, 1).reshape(3, n)
    with Lattice.from_params(dims, dict(P0, rho0=rho0, A=0.0, B=0.0, kappa=0.0), precision=precision) as lat:
        lat.init(np.zeros(n), u0)
        rho, u, _ = lat.moments()
    assert np.abs(rho / rho0 - 1).max() <= tol
    assert np.abs(u - u0).max() <= tol * 0.02 * 5

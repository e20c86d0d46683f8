"""The start in double-float storage is as near to the equilibrium as its
direct sums are: rms errors of f against the FP64 start (itself within 1e-17)
of a tanh interface and of noise around 0.5, 7 points, 20x18x16.  With those
sums they are 1.15e-16 and 1.87e-16 without a flow and 1.30e-16 and 1.94e-16
with one; sums left without renormalising gave 1.47, 1.97, 1.59 and 2.02.  The
bounds lie between.  g is a few 2^-49 of its terms off, whose largest is |phi|:
at most 7.3e-15 and 5.2e-15 were seen, 2^-46 is 1.4e-14."""
import numpy as np
import pytest

from tests.parity import P0

pytestmark = pytest.mark.gpu

DIMS = (20, 18, 16)


@pytest.fixture(scope="module", autouse=True)
def _setup():
    import paper_1405_6162_gb300 as lbpkg
    lbpkg.build()


@pytest.mark.parametrize("start,flow,bound", [("tanh", False, 1.30e-16), ("noise", False, 1.92e-16),
                                              ("tanh", True, 1.45e-16), ("noise", True, 1.98e-16)])
def test_double_float_start(start, flow, bound):
    from paper_1405_6162_gb300 import Lattice
    n = int(np.prod(DIMS))
    x = np.arange(n) % DIMS[0]
    if start == "tanh":
        phi = np.tanh((x - 9.3) / 1.13)
    else:
        phi = 0.5 + 1e-6 * np.random.default_rng(5).uniform(-1, 1, n)
    a = 2 * np.pi * x / DIMS[0]
    u = np.stack([0.003 * np.cos(a + 0.3), 0.01 * np.sin(a + 1.1), 0.02 * np.sin(a)]) if flow else None
    got = {}
    for precision in ("fp64", "fp64_df"):
        with Lattice.from_params(DIMS, P0, precision=precision) as lat:
            lat.init(phi, u)
            got[precision] = lat.get_state()
    f, g = (got["fp64_df"][k] - got["fp64"][k] for k in range(2))
    assert np.sqrt((f * f).mean()) <= bound
    assert np.abs(g).max() <= 2.0 ** -46

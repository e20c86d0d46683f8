"""The wide stencils of a start in float storage, formed by opposite pairs in
FP64, against the FP64 start's: every float within half an ulp of the FP64
value, and the ~2^-46 of the double-float sums behind it, whose terms are at most
1 (as tests/test_gpu_init_moments.py); on smooth and rough fields whose
neighbours all differ, and where extents of 1 and 2 make them one site."""
import numpy as np
import pytest

import lb_inputs as L
from tests.parity import P0

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("points", [19, 27])
@pytest.mark.parametrize("flow", [False, True])
@pytest.mark.parametrize("dims", [(7, 5, 6), (33, 12, 9), (2, 3, 2), (1, 4, 3), (5, 1, 1), (1, 1, 1)])
@pytest.mark.parametrize("smooth", [False, True])
def test_float_start_with_wide_stencils(dims, flow, points, smooth):
    import paper_1405_6162_gb300 as lbpkg
    from paper_1405_6162_gb300 import Lattice
    lbpkg.build()
    n = int(np.prod(dims))
    if smooth:
        z, y, x = np.meshgrid(*(np.arange(k) for k in dims[::-1]), indexing="ij")
        phi = (np.sin(0.9 * x + 0.3) * np.cos(1.1 * y - 0.2) + 0.5 * np.sin(0.7 * z + 0.4 * x)).reshape(-1) * 0.6
    else:
        phi = L.uniform(1300, n, -1, 1)
    u = 0.02 * L.uniform(1301, 3 * n, -1, 1).reshape(3, n) if flow else None
    got = {}
    for precision in ("fp64", "fp32_shifted"):
        with Lattice.from_params(dims, P0, precision=precision) as lat:
            lat.set_stencil(points)
            lat.init(phi, u)
            got[precision] = lat.get_state()
    w = np.array([1 / 3] + [1 / 18] * 6 + [1 / 36] * 12)[:, None] * P0["rho0"]
    for a, b, shift in zip(got["fp32_shifted"], got["fp64"], (w, 0.0)):
        assert (np.abs(a - b) <= 2.0 ** -24 * np.abs(b - shift) + 2.0 ** -44).all()

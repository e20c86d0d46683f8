"""CTA sizes of the two-pass step.  Double-float in every size that
lb_set_kernel takes, with tau_g = 1 (up to 128 threads the collision that
leaves g unread, above the one that reads it) and without: 1e-12 of the oracle,
as every double-float step.  FP32 in the default sizes on either side of their
lines."""
import pytest

import oracle
from tests.parity import P0, TOL_FP64, nonequilibrium_state, rel, to_abi, to_oracle

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("tau_g", [1.0, 0.85])
@pytest.mark.parametrize("rates", [None, (1.3, 0.6)])
@pytest.mark.parametrize("threads", [0, 32, 96, 128, 160, 192, 256])
def test_every_cta_size_matches_oracle(threads, rates, tau_g):
    import paper_1405_6162_gb300 as lbpkg
    from paper_1405_6162_gb300 import Lattice
    lbpkg.build()
    oracle.build()
    dims = (17, 9, 11)
    p = dict(P0, tau=0.7, tau_g=tau_g, kappa=0.06)
    s0 = nonequilibrium_state(dims, p, seed=1100)
    with Lattice.from_params(dims, p, precision="fp64_df") as lat:
        lat.set_kernel("two_pass", threads)
        if rates:
            lat.set_collision("mrt", *rates)
        lat.set_state(*[to_abi(x) for x in s0])
        lat.step(4)
        got = lat.get_state()
    want = oracle.step_mrt(dims, p, *s0, 4, *rates, (0, 0, 0)) if rates else oracle.step(dims, p, *s0, 4)
    for a, w in zip(got, want):
        assert rel(to_oracle(a), w) <= TOL_FP64


# on either side of the FP32 default's lines (24576, 49152, 131072 sites)
@pytest.mark.parametrize("tau_g", [1.0, 0.85])
@pytest.mark.parametrize("dims", [(24, 32, 31), (24, 32, 32), (32, 32, 32), (33, 39, 38), (24, 64, 32), (37, 41, 43),
                                  (64, 64, 32), (51, 51, 51)])
def test_default_cta_sizes_in_fp32_match_oracle(dims, tau_g):
    import paper_1405_6162_gb300 as lbpkg
    from paper_1405_6162_gb300 import Lattice
    lbpkg.build()
    oracle.build()
    p = dict(P0, tau=0.7, tau_g=tau_g, kappa=0.06)
    s0 = nonequilibrium_state(dims, p, seed=1110)
    with Lattice.from_params(dims, p, precision="fp32_shifted") as lat:
        lat.set_state(*[to_abi(x) for x in s0])
        lat.step(3)
        got = lat.get_state()
    for a, w in zip(got, oracle.step(dims, p, *s0, 3)):
        assert rel(to_oracle(a), w) <= 2e-6   # 30 roundings of 6e-8

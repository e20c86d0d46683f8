"""Routes that tau_g = 1 no longer takes: FP32-shifted steps with tau_g != 1 by
every way that leads to them (two passes with 7, 19 and 27 points, the several
rates and a force, the default's bulk kernel on rows of 256 sites), and the
bounded waits of an ensemble's other steps.

Bound.  As in tests/test_gpu_geq.py: 3 steps of a state with |phi| <= 0.5 round
each value about 30 times at 6e-8 of the fields' max-norms: 2e-6."""
import pytest

import oracle
from tests.parity import P0, TOL_FP64, nonequilibrium_state, rel, to_abi, to_oracle

pytestmark = pytest.mark.gpu

TOL_FP32 = 2e-6
P = dict(P0, tau=0.7, tau_g=0.85, kappa=0.06)
FORCE = (1e-5, -2e-5, 3e-5)


@pytest.fixture(scope="module", autouse=True)
def _setup():
    import paper_1405_6162_gb300 as lbpkg
    lbpkg.build()
    oracle.build()


# rows of 256 sites and ny even: the default is the bulk kernel, also where its
# 16 planes a CTA are cut (20 planes) or more than the lattice has
@pytest.mark.parametrize("dims,kernel,npts,rates,force", [
    ((256, 8, 20), "auto", 7, None, (0, 0, 0)), ((256, 2, 5), "auto", 7, None, (0, 0, 0)),
    ((256, 8, 20), "two_pass", 7, None, (0, 0, 0)), ((256, 7, 20), "auto", 7, None, (0, 0, 0)),
    ((33, 18, 21), "auto", 7, None, (0, 0, 0)), ((33, 18, 21), "auto", 19, None, (0, 0, 0)),
    ((33, 18, 21), "auto", 27, None, (0, 0, 0)), ((33, 18, 21), "auto", 7, (1.3, 0.6), FORCE),
    ((33, 18, 21), "auto", 27, (1.7, 0.55), (0, 0, 0)), ((256, 8, 20), "auto", 7, None, FORCE),
    ((128, 96, 90), "auto", 7, None, (0, 0, 0)), ((128, 96, 90), "auto", 19, (1.3, 0.6), FORCE)])
def test_fp32_steps_with_two_rates_match_oracle(dims, kernel, npts, rates, force):
    from paper_1405_6162_gb300 import Lattice
    s0 = nonequilibrium_state(dims, P, seed=1200)
    with Lattice.from_params(dims, P, precision="fp32_shifted") as lat:
        lat.set_kernel(kernel)
        lat.set_stencil(npts)
        if rates:
            lat.set_collision("mrt", *rates)
        lat.set_force(*force)
        lat.set_state(*[to_abi(x) for x in s0])
        lat.step(1)
        lat.step(2)
        got = lat.get_state()
    if npts == 7 and not rates and not any(force):
        want = oracle.step(dims, P, *s0, 3, kind="omp")
    else:
        want = oracle.step_mrt(dims, P, *s0, 3, *(rates or (P["tau"], P["tau"])), force, kind="omp", npts=npts)
    for a, w in zip(got, want):
        assert rel(to_oracle(a), w) <= TOL_FP32


# two passes that read g (tau_g != 1), and the passes that keep moments (tau_g =
# 1, more than 229376 sites); tests/test_gpu_batch.py has those that leave g unread
@pytest.mark.parametrize("tau_g,dims", [(0.85, [(20, 17, 16), (33, 18, 21), (9, 9, 9)]),
                                        (1.0, [(61, 61, 61), (20, 17, 16), (9, 9, 9)])])
@pytest.mark.parametrize("plan", ["lattice", "grid"])
@pytest.mark.parametrize("precision", ["fp64", "fp32_shifted"])
def test_waits_of_the_other_ensemble_steps_are_bounded(precision, plan, tau_g, dims):
    from paper_1405_6162_gb300 import Batch, LBError
    from paper_1405_6162_gb300 import _lib as LL
    specs = [dict(P0, nx=x, ny=y, nz=z, tau=0.8, tau_g=tau_g) for x, y, z in dims]
    start = [nonequilibrium_state(d, P, seed=1210 + k) for k, d in enumerate(dims)]

    def put(b):
        for k, s in enumerate(start):
            b[k].set_state(*[to_abi(x) for x in s])

    with Batch(specs, precision=precision) as b:
        b.set_plan(plan)
        put(b)
        b.run(2)
        b.sync()
        b.set_wait_timeout(0.05)
        LL.check(LL.lib().lb_batch_debug_skip_arrival(b.handle, 1), "hook")
        b.run(3)
        with pytest.raises(LBError) as ei:
            b.sync()
        assert ei.value.code == LL.LB_ERR_TIMEOUT
        LL.check(LL.lib().lb_batch_debug_skip_arrival(b.handle, 0), "hook")
        put(b)
        b.run(1)
        b.run(2)
        b.sync()
        got = [b[k].get_state() for k in range(len(dims))]
    for k, d in enumerate(dims):
        p = {q: specs[k][q] for q in P0}
        for a, w in zip(got[k], oracle.step(d, p, *start[k], 3, kind="omp")):
            assert rel(to_oracle(a), w) <= (TOL_FP64 if precision == "fp64" else TOL_FP32)

"""Steps with tau_g = 1 in the library default: the collision that does not
read g (every precision), and the FP32-shifted steps that keep g as its
equilibrium's moments within one lb_step call.

Bounds.  FP64 and double-float: 1e-12 of the oracle, as every step kernel.
FP32-shifted, per step of a state with |phi| <= 0.5: each of the 38 values is
rounded a few times at 2^-24 of its size, so 3 steps stay within 2e-6 of the
oracle's values (30 roundings of 6e-8), scaled by the fields' max-norms.
The route is a rule on sizes: lattices on both sides of its lines are run, in
one call, split into calls of odd and even length, and with the wide stencils,
the multiple relaxation times and a force.
"""
import numpy as np
import pytest

import lb_inputs as L
import oracle
from tests.parity import P0, TOL_FP64, nonequilibrium_state, rel, to_abi, to_oracle

pytestmark = pytest.mark.gpu

TOL_FP32 = 2e-6
FORCE = (1e-5, -2e-5, 3e-5)
# sites above 2^18 (one row a lane below 2^20 and where ny < 4), short rows, one plane
LARGE = [(65, 64, 64), (31, 97, 90), (128, 128, 64), (700, 3, 250), (13, 150, 140), (600, 500, 1)]
SMALL = [(13, 7, 5), (1, 1, 9), (64, 64, 64), (11, 170, 150)]


@pytest.fixture(scope="module", autouse=True)
def _setup():
    import paper_1405_6162_gb300 as lbpkg
    lbpkg.build()
    oracle.build()


def _run(dims, params, precision, state, calls, npts=7, rates=None, force=(0.0, 0.0, 0.0)):
    from paper_1405_6162_gb300 import Lattice
    with Lattice.from_params(dims, params, precision=precision) as lat:
        lat.set_stencil(npts)
        if rates:
            lat.set_collision("mrt", *rates)
        lat.set_force(*force)
        lat.set_state(to_abi(state[0]), to_abi(state[1]))
        for n in calls:
            lat.step(n)
        return lat.get_state()


def _check(got, want, tol):
    for a, b in zip(got, want):
        assert rel(to_oracle(a), b) <= tol


@pytest.mark.parametrize("calls", [(1,), (2,), (3,), (1, 2)])
@pytest.mark.parametrize("dims", LARGE + SMALL)
def test_fp32_steps_match_oracle(dims, calls):
    p = dict(P0, tau=0.7, kappa=0.06)
    s0 = nonequilibrium_state(dims, p, seed=810)
    want = oracle.step(dims, p, *s0, sum(calls), kind="omp")
    _check(_run(dims, p, "fp32_shifted", s0, calls), want, TOL_FP32)


@pytest.mark.parametrize("npts,rates,force", [(19, None, (0, 0, 0)), (27, (1.3, 0.6), FORCE), (7, (1.7, 0.55), FORCE),
                                              (7, None, FORCE)])
def test_fp32_wide_stencils_rates_and_force(npts, rates, force):
    dims = (65, 64, 64)
    p = dict(P0, tau=0.8, kappa=0.06)
    s0 = nonequilibrium_state(dims, p, seed=820)
    want = oracle.step_mrt(dims, p, *s0, 3, *(rates or (p["tau"], p["tau"])), force, kind="omp", npts=npts)
    _check(_run(dims, p, "fp32_shifted", s0, (3,), npts, rates, force), want, TOL_FP32)


@pytest.mark.parametrize("precision", ["fp64", "fp64_df"])
@pytest.mark.parametrize("tau", [1.0, 0.7])
@pytest.mark.parametrize("dims", [(13, 7, 5), (1, 1, 9), (40, 9, 35)])
def test_unread_g_matches_oracle(dims, tau, precision):
    p = dict(P0, tau=tau, kappa=0.06)
    s0 = nonequilibrium_state(dims, p, seed=830)
    want = oracle.step(dims, p, *s0, 4)
    _check(_run(dims, p, precision, s0, (1, 3)), want, TOL_FP64)


def test_nonfinite_g_is_still_reported():
    """A g that is not finite is not read by the collision, but reaches the
    state through phi."""
    from paper_1405_6162_gb300 import Lattice, LBError
    dims = (65, 64, 64)
    f0, g0 = nonequilibrium_state(dims, P0, seed=840)
    for bad in (np.nan, np.inf):
        g1 = to_abi(g0).copy()
        g1[7, 12345] = bad
        for precision in ("fp64", "fp32_shifted"):
            with Lattice.from_params(dims, P0, precision=precision) as lat:
                lat.set_state(to_abi(f0), g1)
                lat.step(2)
                with pytest.raises(LBError):
                    lat.reduce()


def test_replayed_graph_steps_a_new_start():
    """Steps captured in a CUDA graph depend on nothing but the lattice's
    buffers: after a new start the replay advances that start."""
    import torch
    from paper_1405_6162_gb300 import Lattice
    dims = (65, 64, 64)
    stream = torch.cuda.Stream()
    with torch.cuda.stream(stream), Lattice.from_params(dims, P0, precision="fp32_shifted", stream=stream) as lat:
        phi = [torch.from_numpy(L.spinodal_phi0(*dims, seed=k, amp=0.3)).cuda() for k in (850, 851)]
        lat.init(phi[0])
        lat.step(4)
        stream.synchronize()
        graph = torch.cuda.CUDAGraph()
        lat.init(phi[0])
        with torch.cuda.graph(graph, stream=stream):
            lat.step(4)
        got = []
        for x in phi:
            lat.init(x)
            graph.replay()
            got.append([t.clone() for t in lat.moments(device=True)])
        for x, g in zip(phi, got):
            lat.init(x)
            lat.step(4)
            assert all(torch.equal(a, b) for a, b in zip(lat.moments(device=True), g))
        stream.synchronize()


def test_ensemble_runs_follow_the_members_state():
    """An ensemble's run starts from the members' state, whichever call wrote
    it last: after run(3), a member set to another state (whole or masked) or
    started anew advances that state, and one left alone gives the bits of an
    undivided run."""
    from paper_1405_6162_gb300 import Batch
    specs = [dict(P0, nx=20, ny=17, nz=16, tau=0.8), dict(P0, nx=33, ny=18, nz=21), dict(P0, nx=16, ny=16, nz=40),
             dict(P0, nx=17, ny=31, nz=9, tau=0.6)]
    dims = [(d["nx"], d["ny"], d["nz"]) for d in specs]
    phi = [L.spinodal_phi0(*d, seed=860 + k, amp=0.3) for k, d in enumerate(dims)]
    s1 = [to_abi(x) for x in nonequilibrium_state(dims[1], P0, seed=870)]
    mask = (L.uniform(871, int(np.prod(dims[3])), 0, 1) < 0.4).astype(np.uint8)

    def start(b):
        for k in range(4):
            b[k].init(phi[k])

    with Batch(specs, precision="fp32_shifted") as b, Batch(specs, precision="fp32_shifted") as c:
        start(b)
        start(c)
        b.run(3)
        c.run(3)
        b[1].set_state(*s1)
        b[2].init(phi[2])
        f3, g3 = b[3].get_state_masked(mask)
        b[3].set_state_masked(mask, 1.01 * f3, 0.9 * g3)
        whole3 = b[3].get_state()
        b.run(2)
        got = [b[k].get_state() for k in range(4)]
        # the same from states that no run has touched
        c[0].init(phi[0])
        c[1].set_state(*s1)
        c[2].init(phi[2])
        c[3].set_state(*whole3)
        c.run(2)
        want = [c[k].get_state() for k in range(4)]
        c[0].init(phi[0])
        c.run(5)
        want[0] = c[0].get_state()
    for k in range(4):
        for a, w in zip(got[k], want[k]):
            assert np.array_equal(a, w), k

"""The library default's FP32-shifted steps with tau_g = 1 keep g as its
moments between steps, also between calls: how a run is cut into calls changes
no bit of it, and a call starts from the stored state whichever call wrote it
last.

Bounds.  Cut runs and new starts: equal bits.  After steps of another kernel
or a change of form the state is read back and set on a fresh lattice, which
rounds f once more: 2 steps stay within the 2e-6 of tests/test_gpu_geq.py (30
roundings of 6e-8); moments left from an earlier state are off by its changes,
1e-3 and more.
"""
import numpy as np
import pytest

import lb_inputs as L
from tests.parity import P0, nonequilibrium_state, rel, to_abi

pytestmark = pytest.mark.gpu

TOL_FP32 = 2e-6
P = dict(P0, tau=0.7, kappa=0.06)
FORCE = (1e-5, -2e-5, 3e-5)
# one and two rows a lane (2^20 sites), odd rows, short rows, one plane, few rows
DIMS = [(72, 73, 72), (31, 97, 130), (128, 128, 64), (13, 180, 170), (2049, 1024, 1), (700, 3, 250), (129, 64, 127), (4, 350, 360)]


@pytest.fixture(scope="module", autouse=True)
def _setup():
    import paper_1405_6162_gb300 as lbpkg
    lbpkg.build()


def _lattice(dims, params=P):
    from paper_1405_6162_gb300 import Lattice
    return Lattice.from_params(dims, params, precision="fp32_shifted")


def _state(dims, seed):
    return [to_abi(x) for x in nonequilibrium_state(dims, P, seed=seed)]


@pytest.mark.parametrize("dims,npts,rates,force", [(d, 7, None, (0, 0, 0)) for d in DIMS] + [
    ((72, 73, 72), 19, None, (0, 0, 0)), ((72, 73, 72), 27, (1.3, 0.6), FORCE), ((128, 128, 64), 7, (1.7, 0.55), FORCE)])
def test_bits_do_not_depend_on_the_calls(dims, npts, rates, force):
    start = _state(dims, 900)
    want = None
    for calls in ((6,), (1,) * 6, (2, 4), (3, 1, 2), (5, 1)):
        with _lattice(dims) as lat:
            lat.set_stencil(npts)
            if rates:
                lat.set_collision("mrt", *rates)
            lat.set_force(*force)
            lat.set_state(*start)
            for n in calls:
                lat.step(n)
                lat.reduce()   # watching a run changes nothing either
                lat.moments()
            got = lat.get_state()
        want = want or got
        for a, b in zip(got, want):
            assert np.array_equal(a, b), calls


@pytest.mark.parametrize("dims", [(72, 73, 72), (128, 128, 64)])
@pytest.mark.parametrize("before", [1, 2])
def test_a_new_start_is_followed(dims, before):
    phi = L.spinodal_phi0(*dims, seed=910, amp=0.3)
    s = _state(dims, 911)
    mask = (L.uniform(912, int(np.prod(dims)), 0, 1) < 0.4).astype(np.uint8)

    def masked(lat):
        lat.set_state(*s)
        f, g = lat.get_state_masked(mask)
        lat.set_state_masked(mask, 1.01 * f, 0.9 * g)

    for write in (lambda lat: lat.init(phi), lambda lat: lat.set_state(*s), masked):
        got = []
        for stepped in (True, False):
            with _lattice(dims) as lat:
                if stepped:
                    lat.set_state(*_state(dims, 913))
                    lat.step(before)
                write(lat)
                lat.step(2)
                got.append(lat.get_state())
        for a, b in zip(*got):
            assert np.array_equal(a, b)


def test_a_masked_write_alone_is_followed():
    dims = (72, 73, 72)
    mask = (L.uniform(920, int(np.prod(dims)), 0, 1) < 0.4).astype(np.uint8)
    with _lattice(dims) as lat, _lattice(dims) as fresh:
        lat.set_state(*_state(dims, 921))
        lat.step(3)
        f, g = lat.get_state_masked(mask)
        lat.set_state_masked(mask, f, 0.9 * g)
        fresh.set_state(*lat.get_state())
        for x in (lat, fresh):
            x.step(2)
        for a, b in zip(lat.get_state(), fresh.get_state()):
            assert rel(a, b) <= TOL_FP32


@pytest.mark.parametrize("between", [("two_pass", 0, 0, 0), ("two_pass", 128, 4, 0), ("bulk", 3, 2, 16),
                                     ("fused", 0, 0, 0), ("staged", 0, 0, 0), ("slab", 0, 0, 0), ("lag", 0, 0, 0),
                                     ("taug1", 0, 0, 0)])
@pytest.mark.parametrize("steps", [0, 1, 2])
def test_steps_of_other_kernels_are_followed(between, steps):
    dims = (76, 74, 72)
    with _lattice(dims) as lat, _lattice(dims) as fresh:
        lat.set_state(*_state(dims, 930))
        lat.step(3)
        lat.set_kernel(*between)
        lat.step(steps)
        lat.set_kernel("auto")
        fresh.set_state(*lat.get_state())
        for x in (lat, fresh):
            x.step(2)
        for a, b in zip(lat.get_state(), fresh.get_state()):
            assert rel(a, b) <= TOL_FP32


def test_captured_steps_of_another_kernel_are_followed():
    """Steps of another kernel captured before any default step: their replay
    takes back what the default steps in between left."""
    import torch
    from paper_1405_6162_gb300 import Lattice
    dims = (72, 73, 72)
    stream = torch.cuda.Stream()
    with torch.cuda.stream(stream):
        with Lattice.from_params(dims, P, precision="fp32_shifted", stream=stream) as lat, _lattice(dims) as fresh:
            s = _state(dims, 940)
            for kernel in ("two_pass", "fused"):
                lat.set_kernel(kernel)
                lat.set_state(*s)
                lat.step(2)
                stream.synchronize()
                graph = torch.cuda.CUDAGraph()
                with torch.cuda.graph(graph, stream=stream):
                    lat.step(2)
                lat.set_kernel("auto")
                lat.set_state(*s)
                lat.step(2)
                graph.replay()
                fresh.set_state(*lat.get_state())
                for x in (lat, fresh):
                    x.step(2)
                for a, b in zip(lat.get_state(), fresh.get_state()):
                    assert rel(a, b) <= TOL_FP32
            stream.synchronize()


@pytest.mark.parametrize("launch", [None, (256, 0), (64, 2)])
def test_ensemble_bits_do_not_depend_on_the_runs(launch):
    from paper_1405_6162_gb300 import Batch
    dims = [tuple(int(v) for v in d) for d in np.random.default_rng(950).integers(3, 41, (24, 3))] + [(1, 1, 9), (64, 64, 64)]
    specs = [dict(P0, nx=x, ny=y, nz=z, tau=0.6 + 0.03 * k, kappa=0.02 + 0.002 * k) for k, (x, y, z) in enumerate(dims)]
    start = [_state(d, 951 + k) for k, d in enumerate(dims)]
    want = None
    for runs in ((6,), (1,) * 6, (2, 4), (3, 1, 2)):
        with Batch(specs, precision="fp32_shifted") as b:
            if launch:
                b.set_launch(*launch)
            for k, s in enumerate(start):
                b[k].set_state(*s)
            for n in runs:
                b.run(n)
                b[0].reduce()
            got = [b[k].get_state() for k in range(len(b))]
        want = want or got
        for a, w in zip(got, want):
            assert np.array_equal(a[0], w[0]) and np.array_equal(a[1], w[1]), runs


# on either side of the default's lines: sites, rows and planes that leave
# lanes idle, one plane; and with the wide stencils, several rates and a force
@pytest.mark.parametrize("dims,npts,rates,force", [(d, 7, None, (0, 0, 0)) for d in [
    (70, 70, 70), (72, 72, 72), (4, 330, 360), (4, 350, 360), (2, 700, 700), (1, 900, 900), (128, 5, 600), (130, 6, 600), (600, 2, 500),
    (600, 2, 600), (1024, 1, 512), (1060, 1000, 1), (1024, 1000, 1), (20, 60000, 1), (17, 65000, 1)]] + [
    ((72, 73, 72), 19, None, (0, 0, 0)), ((72, 73, 72), 27, (1.3, 0.6), FORCE), ((4, 350, 360), 27, None, (0, 0, 0)),
    ((72, 73, 72), 7, (1.7, 0.55), FORCE), ((72, 73, 72), 7, None, FORCE)])
def test_default_steps_match_oracle_beside_its_lines(dims, npts, rates, force):
    import oracle
    from tests.parity import to_oracle
    oracle.build()
    s0 = nonequilibrium_state(dims, P, seed=990)
    with _lattice(dims) as lat:
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


def test_an_ensemble_on_many_sites_follows_its_members():
    """A member written between two runs of an ensemble that keeps moments is
    followed, one left alone keeps the bits of an undivided run."""
    from paper_1405_6162_gb300 import Batch
    dims = [(20, 17, 16), (33, 18, 21), (64, 64, 40), (17, 31, 9), (61, 40, 33)]
    specs = [dict(P0, nx=x, ny=y, nz=z, tau=0.6 + 0.1 * k) for k, (x, y, z) in enumerate(dims)]
    start = [_state(d, 960 + k) for k, d in enumerate(dims)]
    other = _state(dims[1], 970)
    phi = L.spinodal_phi0(*dims[2], seed=971, amp=0.3)
    with Batch(specs, precision="fp32_shifted") as b, Batch(specs, precision="fp32_shifted") as c:
        for x in (b, c):
            for k, s in enumerate(start):
                x[k].set_state(*s)
        b.run(3)
        b[1].set_state(*other)
        b[2].init(phi)
        b.run(2)
        got = [b[k].get_state() for k in range(len(dims))]
        c.run(5)
        want = [c[k].get_state() for k in range(len(dims))]
        c[1].set_state(*other)
        c[2].init(phi)
        c.run(2)
        want[1], want[2] = c[1].get_state(), c[2].get_state()
    for k, (a, w) in enumerate(zip(got, want)):
        assert np.array_equal(a[0], w[0]) and np.array_equal(a[1], w[1]), k


# lattices on either side of an ensemble's lines (229376 and 1572864 sites),
# with tau_g = 1 and not, all alike and mixed
@pytest.mark.parametrize("precision,tol", [("fp32_shifted", TOL_FP32), ("fp64", 1e-12)])
@pytest.mark.parametrize("tau_g", [1.0, 0.85, None])
@pytest.mark.parametrize("dims", [[(13, 7, 5), (1, 1, 9), (32, 32, 32), (20, 33, 17)],
                                  [(61, 61, 61), (5, 31, 3), (33, 10, 5)], [(61, 61, 61), (5, 31, 3), (33, 10, 6)],
                                  [(128, 96, 64), (96, 128, 64), (9, 9, 9)]])
def test_ensemble_steps_match_oracle(dims, tau_g, precision, tol):
    import oracle
    from paper_1405_6162_gb300 import Batch
    from tests.parity import to_oracle
    oracle.build()
    specs = [dict(P0, nx=x, ny=y, nz=z, tau=0.7 + 0.1 * k, tau_g=(1.0 if k % 2 else 0.85) if tau_g is None else tau_g)
             for k, (x, y, z) in enumerate(dims)]
    start = [nonequilibrium_state(d, P, seed=980 + k) for k, d in enumerate(dims)]
    with Batch(specs, precision=precision) as b:
        for k, s in enumerate(start):
            b[k].set_state(*[to_abi(x) for x in s])
        b.run(1)
        b.run(2)
        got = [b[k].get_state() for k in range(len(dims))]
    for k, d in enumerate(dims):
        p = {q: specs[k][q] for q in P0}
        for a, w in zip(got[k], oracle.step(d, p, *start[k], 3, kind="omp")):
            assert rel(to_oracle(a), w) <= tol

"""Arguments of ``adjoint.trajectory`` (no GPU): the counts that are refused
before a lattice is made, and the steps that the others take."""
import contextlib

import pytest
import torch

from paper_1405_6162_gb300 import LBError, adjoint

DIMS = (2, 2, 2)


class _Recorder:
    """Stands in for the lattice, the library and the room for states, on the CPU."""

    def __init__(self, monkeypatch):
        self.made, self.steps, self.N, self.handle = 0, [], 8, None
        monkeypatch.setattr(adjoint, "Lattice", self)
        monkeypatch.setattr(adjoint.L, "lib", lambda: self)
        monkeypatch.setattr(adjoint.L, "check", lambda rc, where: None)
        monkeypatch.setattr(adjoint, "_free_bytes", lambda: 1 << 40)
        monkeypatch.setattr(adjoint, "_States", lambda n, count: [(0, 0)] * count)
        monkeypatch.setattr(torch.Tensor, "to", lambda self, **kw: self)

    def from_params(self, *a, **kw):
        self.made += 1
        return self

    def init(self, phi0):
        self.phi0 = phi0

    def step(self, n):
        self.steps.append(n)

    def moments(self, device):
        return None, None, self.phi0.clone()

    def lb_get_state(self, *a):
        return 0


def _trajectory(nsteps, segment, grad):
    phi0 = torch.zeros(8, dtype=torch.float64, requires_grad=True)
    with contextlib.nullcontext() if grad else torch.no_grad():
        return adjoint.trajectory(phi0, torch.tensor(0.04, dtype=torch.float64), DIMS, {}, nsteps, segment)


@pytest.mark.parametrize("grad", [True, False])
@pytest.mark.parametrize("nsteps,segment,error", [(-3, None, ValueError), (-1, 0, ValueError), (200, -1, LBError),
                                                  (1, -7, LBError), (5, 0.5, LBError)])
def test_counts_that_take_no_step_are_refused(monkeypatch, nsteps, segment, error, grad):
    r = _Recorder(monkeypatch)
    with pytest.raises(error):
        _trajectory(nsteps, segment, grad)
    assert r.made == 0


@pytest.mark.parametrize("nsteps,segment,steps", [(0, None, []), (0, 4, []), (0, -1, []), (-3, 2, []), (-3, -2, []),
                                                  (5, None, [1] * 5), (5, 2, [2, 2, 1]), (5, 9, [5])])
def test_segments_take_every_step(monkeypatch, nsteps, segment, steps):
    r = _Recorder(monkeypatch)
    _trajectory(nsteps, segment, True)
    assert r.steps == steps
    r = _Recorder(monkeypatch)
    _trajectory(nsteps, segment, False)
    assert sum(r.steps) == sum(steps)

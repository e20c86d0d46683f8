"""With A = B = kappa = 0 the trajectory is linear in phi0 and a uniform shift of
phi0 shifts phi_T as much, so the gradient of sum_x c(x) phi_T(x) adds up to the
sum of c.  The roundings of a step have either sign and cancel over 1680 sites
and 400 steps; a factor rounded with the same sign in every step adds its 2^-54
(5.6e-17) to the drift each time, so 1e-17 a step tells the two apart."""
import math

import pytest

import lb_inputs as L
from tests.parity import P0

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("tau,tau_g", [(1.0, 1.0), (0.7, 1.0), (1.0, 0.85), (1.3, 1.2)])
def test_gradients_add_up_to_the_weights(tau, tau_g):
    import torch
    import paper_1405_6162_gb300 as lbpkg
    from paper_1405_6162_gb300.adjoint import trajectory
    lbpkg.build()
    dims, steps = (14, 12, 10), 400
    phi = torch.from_numpy(L.spinodal_phi0(*dims, seed=1400, amp=0.3)).cuda().reshape(-1).requires_grad_()
    c = torch.from_numpy(L.uniform(1401, 1680, 0.5, 1.5)).cuda()
    phi_t = trajectory(phi, torch.tensor(0.0, dtype=torch.float64, device="cuda"), dims,
                       dict(P0, tau=tau, tau_g=tau_g, A=0.0, B=0.0, kappa=0.0), steps)
    (g,) = torch.autograd.grad((phi_t * c).sum(), phi)
    total = math.fsum(c.cpu().tolist())
    assert abs(math.fsum(g.cpu().tolist()) / total - 1.0) <= 1e-17 * steps

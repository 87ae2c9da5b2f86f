"""The adjoint at tau = 1, where the collision forgets the populations: the
adjoint field is kept as four values a cell and (FP32) the recorded states as
four moments, with the populations' part of dJ/dtau taken one step earlier.

Against the reverse-mode float64 oracle for J = sum_x w(x) rho(x, T), with the
tolerances of the general adjoint's tests: 1e-9 in FP64, and 2e-3 of the largest
entry (of the value for G and tau) in FP32.  One step (no step after the
last), two, and more than two segments; checkpoints every step; boxes with two
cells, odd sides and rows longer than a warp."""

import numpy as np
import pytest

from oracle import reverse
from paper_1905_09554_gb300 import inputs

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover - CUDA device only
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_1905_09554_gb300 import lbm  # noqa: E402

RL, RV = inputs.COEXISTENCE[("shift", -5.5, 1.0)]


@pytest.mark.parametrize("storage,tol", [("f64", 1e-9), ("f32", 2e-3)])
@pytest.mark.parametrize("box,steps,every", [((12, 12, 20), 1, 1), ((12, 12, 20), 2, 1), ((12, 10, 21), 17, 7),
                                             ((33, 9, 6), 8, 3), ((5, 6, 7), 6, 9), ((2, 3, 4), 5, 2)])
def test_gradient_matches_the_reverse_mode_oracle(box, steps, every, storage, tol):
    nx, ny, nz = box
    rho0 = inputs.noisy_ligament_density(nx, ny, nz, max(1.0, min(nx, ny) / 4), 0.1, RL, RV, 1e-3, seed=31)
    w = 1.0 + np.cos(np.arange(nz) * 2 * np.pi / nz)[:, None, None] + 0.2 * inputs.random_density(nx, ny, nz, seed=3)
    r0 = torch.tensor(rho0, requires_grad=True)
    G, tau = (torch.tensor(v, dtype=torch.float64, requires_grad=True) for v in (-5.5, 1.0))
    (torch.tensor(w) * reverse.rollout(r0, G, tau, steps)).sum().backward()
    with lbm.Lattice(nx, ny, nz, G=-5.5, tau=1.0, storage=storage) as L:
        for _ in range(2):  # the second pass reuses the first one's buffers
            L.adjoint_forward(rho0, steps, every)
            g, gG, gT = L.adjoint_backward(w)
            assert np.abs(g - r0.grad.numpy()).max() <= tol * np.abs(r0.grad.numpy()).max()
            assert abs(gG - G.grad.item()) <= tol * max(abs(G.grad.item()), 1e-6)
            assert abs(gT - tau.grad.item()) <= tol * max(abs(tau.grad.item()), 1e-6)

"""The moment kernels on boxes of every shape, small ones included, which
lbm_step would give to two kernels by itself: the form is asked for, so that
it is the one that runs.

Against single steps of the register-staged population kernel, bit for bit.
Boxes: rows of one pair and a remainder, odd rows (pairs that stick out, stores
value by value), one past a tile, tiles cut in both directions, nz from 1 up;
boxes whose copies hold two sets of fields and such that hold one."""

import numpy as np
import pytest

from oracle import lbm_oracle as o
from oracle import reverse
from paper_1905_09554_gb300 import inputs

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover - CUDA device only
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_1905_09554_gb300 import lbm  # noqa: E402

OPS = {"srt": dict(collision="srt", tau=1.0), "unit": dict(collision="mrt", tau=1.0),
       "paper": dict(collision="mrt", tau=0.8), "shear": dict(collision="mrt", tau=0.8, rates=o.mrt_rates(0.8, rule="shear"))}
WIDE = [(33, 13, 5), (32, 26, 33), (65, 15, 7), (66, 14, 1), (97, 31, 21), (131, 9, 6)]
# rows long enough that the fields fit into a population copy
BOXES = {("f32", "srt"): [(4, 1, 1), (5, 3, 2), (6, 14, 9), *WIDE], ("f32", "unit"): [(4, 1, 1), (5, 3, 2), *WIDE],
         ("f32", "paper"): [(7, 3, 2), (9, 11, 3), *WIDE], ("f32", "shear"): [(6, 14, 9), (7, 3, 2), *WIDE],
         **{(s, op): [(4, 1, 1), (7, 3, 2), (6, 14, 9), *WIDE]
            for s in ("f16", "bf16", "f16l", "bf16l") for op in ("srt", "unit")}}
RL, RV = inputs.COEXISTENCE[("shift", -5.5, 1.0)]


def _state(box, calls, storage, form, **op):
    with lbm.Lattice(*box, G=-5.5, storage=storage, **op) as L:
        L.set_step_forms("one", form)
        if form == "one":
            L.set_kernel_config(kernel=1)
        assert L.step_form(2) == form
        L.set_density(inputs.random_density(*box, seed=7, lo=0.3, hi=1.9))
        for n in calls:
            L.step(n)
        return L.get_populations(), lbm.lbm_current_copy(L.ctx), L.time


@pytest.mark.parametrize("storage,op", list(BOXES))
def test_many_steps_at_once_equal_single_steps(storage, op):
    for box in BOXES[storage, op]:
        for calls in ((2,), (3,), (1, 6, 3)):
            want = _state(box, [1] * sum(calls), storage, "one", **OPS[op])
            got = _state(box, calls, storage, "moments", **OPS[op])
            assert got[1:] == want[1:]
            assert np.array_equal(got[0], want[0]), (box, calls, np.abs(got[0] - want[0]).max())


@pytest.mark.parametrize("box,steps,every", [((12, 12, 20), 1, 1), ((12, 12, 20), 2, 1), ((12, 10, 21), 17, 7),
                                             ((33, 9, 6), 8, 3), ((5, 6, 7), 6, 9), ((4, 1, 1), 5, 2), ((4, 2, 3), 5, 2),
                                             ((70, 15, 8), 5, 2)])
def test_gradient_from_recorded_moments_matches_the_reverse_mode_oracle(box, steps, every):
    """FP32 at tau = 1: the recorded states are moments and the populations' part of dJ/dtau is taken one step
    earlier.  One step (none after the last), two, more than two segments, checkpoints every step, one segment
    longer than the run; sides of one, two and odd cells, more than one tile.  J = sum_x w(x) rho(x, T).

    17 steps of some 200 roundings of 6e-8: 2e-4 of the largest entry; the sums over the box 2e-3, as in the
    general adjoint's tests."""
    nx, ny, nz = box
    rho0 = inputs.noisy_ligament_density(nx, ny, nz, max(1.0, min(nx, ny) / 4), 0.1, RL, RV, 1e-3, seed=31)
    w = 1.0 + np.cos(np.arange(nz) * 2 * np.pi / nz)[:, None, None] + 0.2 * inputs.random_density(nx, ny, nz, seed=3)
    r0 = torch.tensor(rho0, requires_grad=True)
    G, tau = (torch.tensor(v, dtype=torch.float64, requires_grad=True) for v in (-5.5, 1.0))
    (torch.tensor(w) * reverse.rollout(r0, G, tau, steps)).sum().backward()
    with lbm.Lattice(nx, ny, nz, G=-5.5, tau=1.0, storage="f32") as L:
        L.set_step_forms("auto", "moments")
        for _ in range(2):  # the second pass reuses the first one's buffers
            L.adjoint_forward(rho0, steps, every)
            rho = L.density()
            g, gG, gT = L.adjoint_backward(w)
            assert np.abs(g - r0.grad.numpy()).max() <= 2e-4 * np.abs(r0.grad.numpy()).max()
            assert abs(gG - G.grad.item()) <= 2e-3 * max(abs(G.grad.item()), 1e-6)
            assert abs(gT - tau.grad.item()) <= 2e-3 * max(abs(tau.grad.item()), 1e-6)
        L.set_step_forms("auto", "one")
        L.adjoint_forward(rho0, steps, every)  # and the recorded run ends in the bits of the population kernels
        assert np.array_equal(L.density(), rho)


def test_forms_may_change_between_a_recorded_run_and_its_gradient():
    box, w = (33, 9, 6), inputs.random_density(33, 9, 6, seed=3)
    rho0 = inputs.noisy_ligament_density(*box, 2.0, 0.1, RL, RV, 1e-3, seed=31)
    with lbm.Lattice(*box, G=-5.5, tau=1.0, storage="f32") as L:
        got = {}
        for before in ("moments", "one", "two"):
            for after in ("moments", "one", "two"):
                L.set_step_forms("auto", before)
                L.adjoint_forward(rho0, 7, 3)
                L.set_step_forms("one" if after == "one" else "auto", after)
                got[before, after] = L.adjoint_backward(w)
        for (before, _), (g, gG, gT) in got.items():
            ref = got[before, before]
            assert np.array_equal(g, ref[0]) and (gG, gT) == ref[1:], before


@pytest.mark.parametrize("storage", ["f32", "f16", "f64"])
def test_two_kernels_on_a_box_that_steps_in_one_by_itself(storage):
    box = (96, 100, 140)
    want = _state(box, (3,), storage, "one", collision="mrt", tau=0.8)
    got = _state(box, (3,), storage, "two", collision="mrt", tau=0.8)
    assert got[1:] == want[1:] and np.array_equal(got[0], want[0])

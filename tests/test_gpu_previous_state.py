"""After a call of one step the population copy that held the state before it
still does (callers read it there, or take the difference of two states)."""

import numpy as np
import pytest

from oracle import lbm_oracle as o
from paper_1905_09554_gb300 import inputs

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover - CUDA device only
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_1905_09554_gb300 import lbm  # noqa: E402

SHEAR = dict(collision="mrt", tau=0.8, rates=o.mrt_rates(0.8, rule="shear"))


@pytest.mark.parametrize("storage,box,op", [
    ("f64", (33, 20, 12), dict(tau=1.0)), ("f64", (33, 20, 12), dict(tau=0.8)), ("f64", (33, 20, 12), SHEAR),
    ("f64", (96, 90, 200), dict(tau=1.0)),
    ("f32", (33, 20, 12), dict(tau=1.0)), ("f32", (33, 20, 12), dict(collision="mrt", tau=0.8)),
    ("f32", (33, 20, 12), SHEAR), ("f32", (96, 90, 100), dict(tau=1.0)), ("f32", (128, 100, 110), dict(tau=1.0)),
    ("f16", (33, 20, 12), dict(tau=1.0)), ("bf16l", (33, 20, 12), dict(tau=0.9))])
def test_a_call_of_one_step_leaves_the_state_before_it(storage, box, op):
    rho = inputs.random_density(*box, seed=9, lo=0.3, hi=1.9)
    with lbm.Lattice(*box, storage=storage, G=-5.5, kernel=1, **op) as L:
        L.set_density(rho)
        for _ in range(5):
            L.step(1)
        want = L.get_populations()
    with lbm.Lattice(*box, storage=storage, G=-5.5, **op) as L:
        L.set_density(rho)
        for n in (1, 3, 1):
            before = L.stored_populations()
            kept = before.clone()
            L.step(n)
            if n == 1:
                assert L.stored_populations().data_ptr() != before.data_ptr()
                assert not torch.equal(L.stored_populations(), kept)
                assert torch.equal(before, kept)
        assert np.array_equal(L.get_populations(), want)
    # copies that nobody else can read need no second place
    with lbm.Lattice(*box, storage=storage, G=-5.5, torch_buffers=False, **op) as L:
        L.set_density(rho)
        for n in (1, 3, 1):
            L.step(n)
        assert np.array_equal(L.get_populations(), want)


@pytest.mark.parametrize("storage", ["f64", "f32"])
def test_the_first_call_of_one_step_may_be_captured(storage):
    """Two single steps, the first of the context, captured into a graph and replayed three times."""
    box = (33, 20, 12)
    rho = inputs.random_density(*box, seed=9, lo=0.3, hi=1.9)
    with lbm.Lattice(*box, storage=storage, G=-5.5, kernel=1) as L:
        L.set_density(rho)
        for _ in range(6):
            L.step(1)
        want = L.get_populations()
    s = torch.cuda.Stream()
    with torch.cuda.stream(s), lbm.Lattice(*box, storage=storage, G=-5.5) as L:
        assert L.step_form(1) == "two"
        L.set_density(rho)
        s.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=s):
            L.step(1)
            L.step(1)
        for _ in range(3):
            g.replay()
        s.synchronize()
        assert np.array_equal(L.get_populations(), want)

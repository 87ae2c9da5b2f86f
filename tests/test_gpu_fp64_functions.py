"""The FP64 exponential (table-driven) and reciprocal of the step against the
oracle's: one step of a rough field whose densities span four decades, with
rho/rho0 from 1e-3 to far below the smallest normal exp(-rho/rho0), and over
the ends of the exponential's fast range (|rho/rho0| = 700).

One step is about 200 FP64 operations on values up to max(rho, G psi^2): 1e-13
of that is some 500 roundings."""

import numpy as np
import pytest

from oracle import lbm_oracle as o
from paper_1905_09554_gb300 import inputs

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover - CUDA device only
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_1905_09554_gb300 import lbm  # noqa: E402


@pytest.mark.parametrize("kernel", [0, 1])
@pytest.mark.parametrize("rho0", [1.0, 0.05, 5.0 / 700.0, 1e-3])
def test_one_step_over_the_range_of_the_exponential(rho0, kernel):
    rho = 10.0 ** (4.0 * inputs.random_density(33, 7, 9, seed=6, lo=0.0, hi=1.0) - 3.0)
    p = o.Params(G=-1.0, tau=0.9, collision="srt", rho0=rho0)
    f = o.run(o.init_populations(rho), 1, p)
    with lbm.Lattice(33, 7, 9, G=-1.0, tau=0.9, rho0=rho0, storage="f64", kernel=kernel) as L:
        L.set_density(rho)
        L.step(1)
        got = L.moments()[0]
    assert np.abs(got - f.sum(axis=0)).max() <= 1e-13 * max(rho.max(), 1.0)

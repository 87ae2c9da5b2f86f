"""A batch of more boxes than a grid has rows of blocks (65,535)."""

import numpy as np
import pytest

from paper_1905_09554_gb300 import inputs

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover - CUDA device only
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_1905_09554_gb300 import lbm  # noqa: E402


def test_more_boxes_than_a_grid_has_rows():
    """FP32 at tau = 1, two and more steps a call: the first box, those on both sides of the limit and the last
    (the others hold no density) against the same box alone."""
    dims = [(4 + k % 3, 1 + k % 2, 1) for k in range(65540)]
    seen = (0, 1, 65533, 65534, 65535, 65536, 65539)
    rho = {k: inputs.random_density(*dims[k], seed=k, lo=0.3, hi=1.9) for k in seen}
    with lbm.Batch(dims, G=-5.5, tau=1.0, storage="f32") as B:
        for k in seen:
            B.boxes[k].set_density(rho[k])
        B.step(2)
        B.step(3)
        got = {k: B.boxes[k].get_populations() for k in seen}
    for k in seen:
        with lbm.Lattice(*dims[k], G=-5.5, tau=1.0, storage="f32", kernel=1) as L:
            L.set_density(rho[k])
            for _ in range(5):
                L.step(1)
            assert np.array_equal(got[k], L.get_populations()), k

"""A bounded device wait that runs out in a replayed graph is reported, also
when an earlier one has been read (no GPU fault: with test_stall the kernel's
waits give up after about a second and it returns)."""

import pytest

from paper_1905_09554_gb300 import inputs

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover - CUDA device only
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_1905_09554_gb300 import lbm  # noqa: E402


def test_every_replay_that_times_out_is_reported():
    s = torch.cuda.Stream()
    with torch.cuda.stream(s), lbm.Lattice(32, 16, 8, storage="f32", kernel=4, tile_y=16, test_stall=1) as L:
        L.set_density(inputs.random_density(32, 16, 8, seed=3))
        s.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=s):
            L.step(1)
        L.set_kernel_config(kernel=1)  # the graph keeps the kernel that it captured
        for _ in range(2):
            g.replay()
            with pytest.raises(lbm.LbmError, match="LBM_ETIMEOUT"):
                L.diag(2.0, 0.1)
            L.diag(2.0, 0.1, raise_nonfinite=False)  # the error word was cleared

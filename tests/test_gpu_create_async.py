"""Creating a context does not wait for what the caller has enqueued on its
stream."""

import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover - CUDA device only
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_1905_09554_gb300 import lbm  # noqa: E402


@pytest.mark.parametrize("storage,box", [("f32", (64, 64, 144)), ("f16l", (64, 64, 200)), ("f64", (32, 32, 64))])
def test_creation_returns_while_the_stream_is_busy(storage, box):
    with lbm.Lattice(*box, storage=storage):  # kernels loaded, allocator warm
        pass
    torch.cuda.synchronize()
    done = torch.cuda.Event()
    torch.cuda._sleep(400_000_000)  # some 0.2 s on the current stream
    done.record()
    L = lbm.Lattice(*box, storage=storage)
    busy = not done.query()
    L.close()
    assert busy

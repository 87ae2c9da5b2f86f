"""lbm_diag_noalloc gives the bits of lbm_diag, whether a slice is summed in one
part or in several.  The file is named so that pytest collects it late."""

import ctypes

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover - CUDA device only
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_1905_09554_gb300 import inputs, lbm  # noqa: E402


@pytest.mark.parametrize("storage", ["f64", "f32", "f16", "bf16"])
@pytest.mark.parametrize("box", [(5, 3, 2), (48, 40, 72), (64, 33, 9), (97, 85, 13), (200, 150, 40)])
def test_both_diagnostics_have_the_same_bits(box, storage):
    nx, ny, nz = box
    with lbm.Lattice(nx, ny, nz, storage=storage) as L:
        L.set_density(inputs.random_density(nx, ny, nz, seed=2, lo=0.3, hi=1.9))
        L.step(2)
        ref = L.diag(2.0, 0.1)
        m, mo = ctypes.c_double(), (ctypes.c_double * 3)()
        area, mx = np.empty(nz), np.empty(nz)
        st = lbm.lbm_diag_noalloc(L.stored_populations().data_ptr(), lbm.STORAGE[storage], nx, ny, nz, 1.0, 1.0, 2.0,
                                  0.1, ctypes.addressof(m), ctypes.addressof(mo), area.ctypes.data, mx.ctypes.data, 0,
                                  torch.cuda.current_stream().cuda_stream)
    assert st == lbm.LBM_OK
    assert m.value == ref["mass"] and np.array_equal(mo[:], ref["mom"])
    assert np.array_equal(area, ref["area_z"]) and np.array_equal(mx, ref["maxrho_z"])

"""The FP64 exponential and reciprocal of the step (csrc/collide.cuh) against
64-bit-mantissa (or wider) values, argument by argument: a small program that
calls the two device functions, compiled here.

The exponential's last operation is one rounded sum of a table entry and a
term below 0.011, whose own roundings, the polynomial's and the tables' second
words add less than 0.03 ulp: 0.55 ulp.  It may not be worse than exp either.
The reciprocal has the bits of the division."""

import ctypes
import os
import shutil
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover - CUDA device only
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_1905_09554_gb300 import build  # noqa: E402

SOURCE = r"""
#include "collide.cuh"
__global__ void values(const double* a, const double* x, double* out, int n) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    out[i] = lbm::exp_table(a[i]);
    out[n + i] = exp(a[i]);
    out[2 * n + i] = lbm::recip<double>(x[i]);
    out[3 * n + i] = 1.0 / x[i];
}
// x force of a random neighbourhood (4 numbers a cell: psi and the sums of its planes) at strength G
__global__ void forces(const double* v, double* out, int n, const __grid_constant__ lbm::StepArgs a) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    lbm::PsiView<double> lo{}, mid{}, hi{};
    mid.c = v[i];
    mid.ex = v[n + i];
    mid.dx = v[2 * n + i];
    lo.ex = v[3 * n + i];
    const lbm::Force<double> F = lbm::force_of(lo, mid, hi, lbm::par<double>(a.gw, a.gwf));
    out[i] = F.g;
    out[n + i] = F.sx;
}
extern "C" int force(const double* v, double* out, int n, double G) {
    lbm::StepArgs a{};
    a.G = G;
    lbm::round_params(a);
    forces<<<(n + 255) / 256, 256>>>(v, out, n, a);
    return cudaDeviceSynchronize();
}
extern "C" int run(const double* a, const double* x, double* out, int n) {
    values<<<(n + 255) / 256, 256>>>(a, x, out, n);
    return cudaDeviceSynchronize();
}
"""


@pytest.fixture(scope="module")
def values(tmp_path_factory):
    if np.finfo(np.longdouble).nmant < 63:
        pytest.skip("no wider host type")
    if not (shutil.which("nvcc") or os.path.exists("/usr/local/cuda/bin/nvcc")):
        pytest.skip("no nvcc")
    d = tmp_path_factory.mktemp("fp64")
    (d / "values.cu").write_text(SOURCE)
    lib = str(d / "values.so")
    subprocess.run([build.nvcc(), *build.FLAGS, *build.ARCH, "-I" + build.CSRC, "-shared", "-o", lib,
                    str(d / "values.cu")], check=True)
    run, force = ctypes.CDLL(lib).run, ctypes.CDLL(lib).force

    def forces(v, G):
        tv = torch.tensor(v, dtype=torch.float64, device="cuda")
        out = torch.empty(2 * v.shape[1], dtype=torch.float64, device="cuda")
        torch.cuda.synchronize()
        assert force(ctypes.c_void_p(tv.data_ptr()), ctypes.c_void_p(out.data_ptr()), v.shape[1], ctypes.c_double(G)) == 0
        return out.cpu().numpy().reshape(2, -1)

    def call(a, x):
        n = len(a)
        ta, tx = (torch.tensor(v, dtype=torch.float64, device="cuda") for v in (a, x))
        out = torch.empty(4 * n, dtype=torch.float64, device="cuda")
        torch.cuda.synchronize()
        assert run(*(ctypes.c_void_p(t.data_ptr()) for t in (ta, tx, out)), n) == 0
        return out.cpu().numpy().reshape(4, n)

    call.forces = forces
    return call


def _ulps(v, want):
    return np.abs((v.astype(np.longdouble) - want) / np.spacing(want.astype(np.float64)))


def test_exponential_rounds_as_well_as_exp(values):
    rng = np.random.default_rng(5)
    n = 1 << 16
    # densities of a two-phase state, the whole fast range, and steps of ln2/64 (the ends of the table's intervals)
    k = rng.integers(-64 * 9, 1, n)
    a = np.concatenate([-4.6 * rng.random(n), 1380.0 * rng.random(n) - 690.0,
                        (k + 0.5) * np.log(2.0) / 64 * (1 + 1e-12 * rng.standard_normal(n)),
                        k * np.log(2.0) / 64 - 1e-9 * rng.random(n)])
    got, ref = values(a, np.ones_like(a))[:2]
    want = np.exp(a.astype(np.longdouble))
    assert _ulps(got, want).max() <= 0.55
    assert _ulps(got, want).max() <= _ulps(ref, want).max()


def test_ends_of_the_exponentials_fast_range(values):
    a = np.array([0.0, -0.0, -699.9999, -700.0, -700.0001, -745.2, -1e5, 699.9999, 700.0, 709.0, 1e4, np.inf, -np.inf,
                  np.nan])
    got, ref = values(a, np.ones_like(a))[:2]
    with np.errstate(over="ignore", under="ignore"):
        near = np.nextafter(ref, np.inf), ref, np.nextafter(ref, -np.inf)
    assert all(any(np.array_equal([g], [v], equal_nan=True) for v in row) for g, row in zip(got, zip(*near)))


def test_reciprocal_has_the_bits_of_the_division(values):
    rng = np.random.default_rng(6)
    n = 1 << 17
    x = np.concatenate([0.02 + 3.0 * rng.random(n), np.ldexp(1.0 + rng.random(n), rng.integers(-300, 300, n)),
                        [0.0, -0.0, np.inf, -np.inf, np.nan, 5e-324, 1e-310, 2.0 ** -1022, 1.7976931348623157e308, 1.0,
                         -3.0, 2.0 - 2.0 ** -52, 1.0 + 2.0 ** -52, -1e-300]])
    inv, div = values(np.zeros_like(x), x)[2:]
    assert np.array_equal(inv, div, equal_nan=True)


@pytest.mark.parametrize("G", [-5.5, -5.3, -7.0, -4.9])
def test_force_weight_rounds_as_the_equilibriums(values, G):
    """The force carries the rounded weight 1/36 of w rho as a factor of its own, bit for bit: -G/36 rounded in one
    would be off from it by a common factor of up to 1.7e-16 in every cell."""
    rng = np.random.default_rng(8)
    v = rng.random((4, 1 << 16)) + 0.05
    g, sx = values.forces(v, G)
    assert np.array_equal(g, (-G * v[0]) * (1.0 / 36.0))
    assert np.abs(sx - (2 * v[1] + v[2] + v[3])).max() <= 4e-15

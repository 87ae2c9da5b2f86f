"""Calls of several steps go through the moment fields where the collision
forgets the other populations (SRT at tau = 1; MRT whose rates outside
{e, 3pxx, pww, pxy, pyz, pxz} are 1).  They must leave exactly the populations
that single steps of the register-staged population kernel leave.

Boxes: smaller than a tile, odd and ragged sides, one past a tile, a box whose
rows are shorter than two tiles apart, nz from 1 up; even and odd numbers of
steps (the state ends in the copy that single steps would use)."""

import numpy as np
import pytest

from oracle import lbm_oracle as o
from paper_1905_09554_gb300 import inputs

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover - CUDA device only
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_1905_09554_gb300 import lbm  # noqa: E402

OPS = {"srt": dict(collision="srt", tau=1.0), "unit": dict(collision="mrt", tau=1.0),
       "paper": dict(collision="mrt", tau=0.8), "shear": dict(collision="mrt", tau=0.8, rates=o.mrt_rates(0.8, rule="shear"))}
BOXES = [(4, 1, 1), (5, 3, 2), (6, 14, 9), (33, 13, 5), (32, 26, 33), (65, 15, 7), (97, 31, 21), (128, 40, 130)]


def _state(box, kernel, calls, storage="f32", **op):
    nx, ny, nz = box
    rho = inputs.random_density(nx, ny, nz, seed=7, lo=0.3, hi=1.9)
    with lbm.Lattice(nx, ny, nz, G=-5.5, storage=storage, kernel=kernel, **op) as L:
        L.set_density(rho)
        for n in calls:
            L.step(n)
        return L.get_populations(), lbm.lbm_current_copy(L.ctx), L.time


@pytest.mark.parametrize("op", list(OPS))
@pytest.mark.parametrize("box", BOXES)
def test_many_steps_at_once_equal_single_steps(box, op):
    for calls in ((2,), (3,), (1, 6, 3)):
        want, copy, t = _state(box, 1, [1] * sum(calls), **OPS[op])
        got, copy2, t2 = _state(box, 0, calls, **OPS[op])
        assert (copy, t) == (copy2, t2)
        assert np.array_equal(got, want), (calls, np.abs(got - want).max())


@pytest.mark.parametrize("storage", ["f16", "bf16", "f16l", "bf16l"])
@pytest.mark.parametrize("op", ["srt", "unit"])
def test_16_bit_storage_is_rounded_at_every_step(storage, op):
    """The populations between the steps of one call go through the storage's rounding too: same bits."""
    for box in ((32, 26, 33), (6, 14, 9), (65, 15, 7), (130, 9, 5)):
        for calls in ((2,), (1, 6, 3)):
            want, _, _ = _state(box, 1, [1] * sum(calls), storage, **OPS[op])
            got, _, _ = _state(box, 0, calls, storage, **OPS[op])
            assert np.array_equal(got, want), (box, calls, np.abs(got - want).max())


@pytest.mark.parametrize("op", list(OPS))
def test_batches_at_once_equal_single_steps(op):
    """Every box of a batch against the same box alone on the register-staged kernel; one box has rows too
    short for two sets of fields in a population copy."""
    dims = [(32, 26, 33), (5, 3, 2), (64, 14, 20), (97, 31, 21), (48, 48, 7)]
    rho = [inputs.random_density(*d, seed=30 + k, lo=0.3, hi=1.9) for k, d in enumerate(dims)]
    with lbm.Batch(dims, G=-5.5, storage="f32", **OPS[op]) as B:
        for v, r in zip(B.boxes, rho):
            v.set_density(r)
        for n in (1, 4, 3):
            B.step(n)
        got = [v.get_populations() for v in B.boxes]
    for d, r, f in zip(dims, rho, got):
        with lbm.Lattice(*d, G=-5.5, storage="f32", kernel=1, **OPS[op]) as L:
            L.set_density(r)
            for _ in range(8):
                L.step(1)
            assert np.array_equal(f, L.get_populations()), d


@pytest.mark.parametrize("op", ["srt", "unit", "paper", "shear", "srt09", "general"])
def test_two_kernel_fp64_step_is_bit_identical(op):
    """FP64 steps in two kernels (in place where the moments suffice, through a psi field otherwise) against
    the register-staged kernel, single lattices and batches."""
    more = {"srt09": dict(collision="srt", tau=0.9),
            "general": dict(collision="mrt", tau=0.9, rates=[0.8 + 0.04 * ((7 * k) % 19) for k in range(19)])}
    kw = dict(OPS, **more)[op]
    boxes = [(1, 1, 5), (2, 3, 2), (33, 13, 5), (65, 15, 7), (32, 32, 64)]
    want = []
    for box in boxes:
        f, copy, t = _state(box, 1, [1] * 7, "f64", **kw)
        got, copy2, t2 = _state(box, 0, (2, 5), "f64", **kw)
        assert (copy, t) == (copy2, t2)
        assert np.array_equal(got, f), box
        want.append(f)
    with lbm.Batch(boxes, G=-5.5, storage="f64", **kw) as B:
        for v, d in zip(B.boxes, boxes):
            v.set_density(inputs.random_density(*d, seed=7, lo=0.3, hi=1.9))
        for n in (3, 4):
            B.step(n)
        for v, f in zip(B.boxes, want):
            assert np.array_equal(v.get_populations(), f), v.shape


@pytest.mark.parametrize("op", list(OPS))
def test_spans_that_end_within_tiles_and_boxes(op):
    """More tiles than the device has blocks: a block's span of planes ends within a tile and goes on in the
    next one, or in the next box of a batch."""
    box = (256, 620, 7)
    want, _, _ = _state(box, 1, [1] * 3, **OPS[op])
    got, _, _ = _state(box, 0, (3,), **OPS[op])
    assert np.array_equal(got, want), np.abs(got - want).max()
    dims = [(70, 27, 3 + k % 7) for k in range(60)]
    with lbm.Batch(dims, G=-5.5, storage="f32", **OPS[op]) as B:
        for v, d in zip(B.boxes, dims):
            v.set_density(inputs.random_density(*d, seed=7, lo=0.3, hi=1.9))
        B.step(3)
        got = [v.get_populations() for v in B.boxes]
    for d in dims[:7]:
        want, _, _ = _state(d, 1, [1] * 3, **OPS[op])
        for k, f in enumerate(got):
            if dims[k] == d:
                assert np.array_equal(f, want), (k, d)


@pytest.mark.parametrize("storage,op", [("f32", "srt09"), ("f32", "general"), ("f32", "srt"), ("f16", "srt09"),
                                        ("bf16", "general"), ("f16l", "srt09"), ("bf16l", "paper")])
def test_two_kernel_step_of_small_boxes_is_bit_identical(storage, op):
    """FP32 and 16-bit boxes that step in two kernels, against the register-staged kernel: fewer cells than a
    block has threads, one more, a last block that is nearly empty, odd and even rows."""
    more = {"srt09": dict(collision="srt", tau=0.9),
            "general": dict(collision="mrt", tau=0.9, rates=[0.8 + 0.04 * ((7 * k) % 19) for k in range(19)])}
    kw = dict(OPS, **more)[op]
    for box in ((1, 3, 5), (257, 1, 1), (32, 8, 2), (33, 13, 5), (64, 50, 31), (101, 99, 97)):
        want, copy, t = _state(box, 1, [1] * 3, storage, **kw)
        got, copy2, t2 = _state(box, 0, [1] * 3, storage, **kw)
        assert (copy, t) == (copy2, t2)
        assert np.array_equal(got, want), (box, np.abs(got - want).max())

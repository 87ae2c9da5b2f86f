"""The forms a call of lbm_step takes (one kernel, two kernels, moments between
the steps): a kernel or launch shape that was asked for is the one that steps,
the tuner times what steps and keeps the fastest, and its cache restores it."""

import json

import numpy as np
import pytest

from oracle import lbm_oracle as o
from paper_1905_09554_gb300 import inputs

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover - CUDA device only
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_1905_09554_gb300 import lbm  # noqa: E402

# (storage, box, tau, automatic forms of step(1) and step(n))
CASES = [("f64", (33, 20, 12), 0.8, ("two", "two")), ("f64", (32, 32, 64), 1.0, ("two", "two")),
         ("f32", (64, 40, 30), 0.8, ("two", "two")), ("f32", (64, 64, 144), 1.0, ("two", "moments")),
         ("f32", (128, 128, 130), 1.0, ("one", "moments")), ("f32", (128, 128, 130), 0.8, ("one", "one")),
         ("f16", (97, 85, 31), 0.9, ("two", "two")), ("f16l", (48, 36, 20), 0.8, ("two", "two"))]


def _populations(L, rho, calls=(1, 4, 1)):
    L.set_density(rho)
    for n in calls:
        L.step(n)
    return L.get_populations()


def _forms(L):
    return L.step_form(1), L.step_form(5)


@pytest.mark.parametrize("storage,box,tau,forms", CASES)
def test_a_shape_that_was_asked_for_steps(storage, box, tau, forms):
    rho = inputs.random_density(*box, seed=9, lo=0.3, hi=1.9)
    kw = dict(storage=storage, tau=tau, G=-5.5)
    with lbm.Lattice(*box, kernel=1, **kw) as L:
        assert _forms(L) == ("one", "one")
        want = _populations(L, rho)
    with lbm.Lattice(*box, **kw) as L:
        assert _forms(L) == forms
        assert np.array_equal(_populations(L, rho), want)
        kernel = L.kernel_config()["kernel"]
        L.set_kernel_config(kernel, 8, 4)
        assert _forms(L) == ("one", "one")
        assert L.kernel_config()["tile_y"] == 8
        assert np.array_equal(_populations(L, rho), want)
        L.set_kernel_config()
        assert _forms(L) == forms
    for shape in (dict(tile_y=8), dict(zchunk=5)):
        with lbm.Lattice(*box, **shape, **kw) as L:
            assert _forms(L) == ("one", "one")
            assert np.array_equal(_populations(L, rho), want)


@pytest.mark.parametrize("storage,box,tau,forms", CASES)
def test_the_tuner_times_the_forms_and_its_cache_restores_them(storage, box, tau, forms, tmp_path):
    rho = inputs.random_density(*box, seed=9, lo=0.3, hi=1.9)
    kw = dict(storage=storage, tau=tau, G=-5.5)
    path = str(tmp_path / "tune.json")
    with lbm.Lattice(*box, kernel=1, **kw) as L:
        want = _populations(L, rho)
    with lbm.Lattice(*box, **kw) as L:
        pick = L.tune(trial_steps=2, cache=path)
        tuned, many = _forms(L), L.step_form(10 ** 6)
        assert (tuned[0], many) == tuple(pick["forms"][:2])
        assert L.step_form(pick["forms"][2]) == many
        assert np.array_equal(_populations(L, rho), want)
        L.set_step_forms("one", "one")  # the shape that was found fastest, whatever won
        assert np.array_equal(_populations(L, rho), want)
    with lbm.Lattice(*box, **kw) as L:
        again = L.tune(trial_steps=2, cache=path)
        assert again["cached"] and again["forms"] == pick["forms"]
        assert (L.step_form(1), L.step_form(pick["forms"][2]), L.step_form(10 ** 6)) == (tuned[0], many, many)
    data = json.load(open(path))
    for entry in data.values():  # as stored before there were forms
        del entry["forms"]
    json.dump(data, open(path, "w"))
    with lbm.Lattice(*box, **kw) as L:
        assert L.tune(trial_steps=2, cache=path)["cached"]
        assert _forms(L) == ("one", "one")


def test_the_tuner_finds_two_kernels_and_moments_where_they_are_several_times_faster():
    with lbm.Lattice(32, 32, 64, storage="f64") as L:  # 8.1 against 1.1 ms per 50 steps
        assert L.tune()["forms"] == ["two", "two", 2]
    with lbm.Lattice(256, 256, 300, storage="f32") as L:  # 56 against 23 ms per 50 steps of twice the box
        assert L.tune()["forms"][:2] == ["one", "moments"]


def test_forms_that_cannot_serve_are_refused():
    with lbm.Lattice(16, 8, 8, tau=0.8, storage="f32") as L:
        before = _forms(L)
        with pytest.raises(lbm.LbmError, match="LBM_EUNSUPPORTED"):
            L.set_step_forms("one", "moments")  # SRT off tau = 1 keeps all populations
        assert lbm.lbm_set_step_forms(L.ctx, 3, 0) == lbm.LBM_EINVAL  # moments between the steps of one step
        assert lbm.lbm_set_step_forms(L.ctx, 0, 4) == lbm.LBM_EINVAL
        assert _forms(L) == before
        assert lbm.lbm_step_form(L.ctx, 0) == 0
    with lbm.Lattice(3, 8, 8, storage="f32") as L:
        with pytest.raises(lbm.LbmError, match="LBM_EUNSUPPORTED"):
            L.set_step_forms("auto", "moments")  # rows of fewer than 4 cells
    with lbm.Lattice(16, 8, 8, G=-7.0, G2=1.5, storage="f32") as L:
        assert _forms(L) == ("one", "one")
        with pytest.raises(lbm.LbmError, match="LBM_EUNSUPPORTED"):
            L.set_step_forms("two", "two")
    with lbm.Batch([(8, 8, 8)], storage="f32") as B:
        with pytest.raises(lbm.LbmError, match="LBM_EINVAL"):
            B.boxes[0].set_step_forms("one", "one")


DIMS = [(32, 32, 50), (20, 17, 33), (48, 48, 75), (33, 40, 9), (64, 64, 101)]


@pytest.mark.parametrize("storage,tau,forms", [("f64", 1.0, ("two", "two")), ("f64", 0.9, ("one", "one")),
                                               ("f32", 1.0, ("one", "moments")), ("f32", 0.9, ("one", "one"))])
def test_batches_step_by_a_shape_that_was_asked_for_and_their_tuner_times_the_forms(storage, tau, forms, tmp_path):
    rho = [inputs.random_density(*d, seed=30 + k, lo=0.3, hi=1.9) for k, d in enumerate(DIMS)]
    path = str(tmp_path / "tune.json")

    def populations(B):
        for v, r in zip(B.boxes, rho):
            v.set_density(r)
        for n in (1, 4, 3, 2):
            B.step(n)
        return [v.get_populations() for v in B.boxes]

    kw = dict(storage=storage, tau=tau, G=-5.5)
    with lbm.Batch(DIMS, tile_y=8, zchunk=16, **kw) as B:
        assert (B.step_form(1), B.step_form(2)) == ("one", "one") == (B.boxes[0].step_form(1), B.boxes[0].step_form(2))
        want = populations(B)
    with lbm.Batch(DIMS, **kw) as B:
        assert (B.step_form(1), B.step_form(12)) == forms
        assert all(np.array_equal(a, b) for a, b in zip(populations(B), want))
        B.set_step_forms("one", "one")  # the graphs of the other form are gone
        assert all(np.array_equal(a, b) for a, b in zip(populations(B), want))
        B.set_step_forms()
        assert (B.step_form(1), B.step_form(12)) == forms
        if forms[1] != "moments":
            with pytest.raises(lbm.LbmError, match="LBM_EUNSUPPORTED"):
                B.set_step_forms("auto", "moments")
    with lbm.Batch(DIMS, tune_cache=path, **kw) as B:
        tuned = B.step_form(1), B.step_form(2), B.step_form(10 ** 6)
        assert all(np.array_equal(a, b) for a, b in zip(populations(B), want))
    if storage == "f64":  # several times faster wherever it can run
        assert tuned[:2] == forms
    entry, = json.load(open(path)).values()
    assert tuple(entry["forms"][:2]) == (tuned[0], tuned[2])
    with lbm.Batch(DIMS, tune_cache=path, **kw) as B:
        assert (B.step_form(1), B.step_form(2), B.step_form(10 ** 6)) == tuned
        assert all(np.array_equal(a, b) for a, b in zip(populations(B), want))


PAPER, SHEAR = dict(collision="mrt", tau=0.9), dict(collision="mrt", tau=0.9, rates=o.mrt_rates(0.9, rule="shear"))


@pytest.mark.parametrize("box,op,n,form", [
    # us a call through moments / in single steps: 607 / 780, 950 / 808; 1051 / 800, 1355 / 1200, 1520 + / 2000;
    # 800 / 798, 1130 / 1197
    ((256, 256, 200), dict(tau=1.0), 2, "moments"), ((255, 255, 200), dict(tau=1.0), 2, "one"),
    ((255, 255, 200), dict(tau=1.0), 5, "moments"), ((256, 256, 200), PAPER, 2, "one"), ((256, 256, 200), PAPER, 3, "one"),
    ((256, 256, 200), PAPER, 20, "moments"), ((256, 256, 200), SHEAR, 2, "one"), ((256, 256, 200), SHEAR, 5, "moments"),
    ((160, 150, 200), PAPER, 5, "one"), ((128, 128, 128), dict(tau=1.0), 2, "moments")])
def test_short_calls_go_through_moments_only_where_that_makes_up_for_its_ends(box, op, n, form):
    with lbm.Lattice(*box, storage="f32", G=-5.5, **op) as L:
        assert L.step_form(n) == form
        L.set_step_forms("one", "moments", 7)
        assert [L.step_form(k) for k in (1, 2, 6, 7, 8)] == ["one"] * 3 + ["moments"] * 2


def test_batches_of_narrow_boxes_do_not_go_through_ten_moments():
    """24 boxes of 32 x 32, us a step: 94 with 10 moments, 80 in one kernel; 59 with 4, 69 in one kernel."""
    dims = [(32, 32, 40 + 3 * k) for k in range(24)]
    with lbm.Batch(dims, storage="f32", G=-5.5, **PAPER) as B:
        assert [B.step_form(n) for n in (1, 2, 50)] == ["one"] * 3
    with lbm.Batch(dims, storage="f32", G=-5.5, tau=1.0) as B:
        assert [B.step_form(n) for n in (1, 2, 50)] == ["one", "one", "moments"]

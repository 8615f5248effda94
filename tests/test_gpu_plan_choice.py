"""A launch plan that is set or tuned is the one that runs, whatever the batch: at 256^2 and 512^2 in
complex64, where a few fields have a default plan of their own.  A field's values under one plan are
the same bits in every batch, so those of a larger batch show which plan ran."""
import json

import numpy as np
import pytest

import kd_inputs as I
from oracle import kd_oracle as O

pytestmark = pytest.mark.gpu

# side, the default plan of many fields, fields with and without a plan of their own
SIDES = [(256, (6, 0), 3, 7), (512, (5, 9), 2, 5)]


@pytest.fixture(scope="module")
def kd():
    import torch
    import __graft_entry__
    __graft_entry__.build()
    import paper_1902_00387_gb300 as kd
    kd.load()
    torch.cuda.init()
    return kd


def context(kd, n):
    return kd.kd_create(kd.make_params(O.GALLOWAY_PROCTOR, n, 0.57, 1e3, 0.64 / n, kd.KD_C64))


def steps(kd, ctx, n, fields):
    import torch
    x = torch.tensor(I.initial_batch(n, 0.57, range(fields)), dtype=torch.complex64, device="cuda")
    y = torch.empty_like(x)
    kd.kd_fine_batched(ctx, x, y, torch.arange(fields, dtype=torch.float64, device="cuda"), 2, fields)
    torch.cuda.synchronize()
    return y.cpu().numpy()


@pytest.mark.parametrize("n,plan,few,many", SIDES)
def test_the_default_plan_can_be_chosen_for_a_few_fields(kd, n, plan, few, many):
    ctx = context(kd, n)
    try:
        assert kd.kd_get_plan(ctx, kd.KD_GRID_FINE) == plan
        ref, own = steps(kd, ctx, n, many)[:few], steps(kd, ctx, n, few)
        assert not np.array_equal(own, ref)                     # few fields have other kernels
        kd.kd_set_plan(ctx, kd.KD_GRID_COARSE, 0, 0)            # says nothing about the fine grid
        assert np.array_equal(steps(kd, ctx, n, few), own)
        kd.kd_set_plan(ctx, kd.KD_GRID_FINE, *plan)
        assert np.array_equal(steps(kd, ctx, n, few), ref)
        assert np.array_equal(steps(kd, ctx, n, many)[:few], ref)
    finally:
        kd.kd_destroy(ctx)


@pytest.mark.parametrize("n,plan,few,many", SIDES)
def test_a_tuned_plan_runs(kd, n, plan, few, many, tmp_path):
    import torch
    ctx = context(kd, n)
    try:
        ref = steps(kd, ctx, n, many)[:few]
        cache = tmp_path / "tune.json"
        cache.write_text(json.dumps({"kd_autotune": 1, "entries": [
            {"device": torch.cuda.get_device_name(0), "n": n, "prec": 0, "batch": 4 if few == 3 else 2,
             "col": plan[0], "row": plan[1], "ms_per_step": 0.1}]}))
        assert kd.kd_autotune(ctx, kd.KD_GRID_FINE, few, 1, str(cache)) == -1.0
        assert np.array_equal(steps(kd, ctx, n, few), ref)
    finally:
        kd.kd_destroy(ctx)


def test_a_serial_run_chooses_nothing(kd):
    n, few = 256, 3
    ctx = context(kd, n)
    try:
        own = steps(kd, ctx, n, few)
        u = np.zeros((2, 3, n, n), np.complex128)
        kd.kd_fine_serial(ctx, I.initial_field(n, 0.57, 1), 1.28 / n, 1, u)
        assert kd.kd_get_plan(ctx, kd.KD_GRID_FINE) == (6, 0)
        assert np.array_equal(steps(kd, ctx, n, few), own)
    finally:
        kd.kd_destroy(ctx)

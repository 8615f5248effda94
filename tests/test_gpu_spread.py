"""complex128 kept sets on 192 points: a few fields step by launches over the whole GPU, more in
clusters, with the same bits; and the smallest sets on 16 points."""
import numpy as np
import pytest

import kd_inputs as I
from oracle import kd_oracle as O

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def kd():
    import torch
    import __graft_entry__
    __graft_entry__.build()
    import paper_1902_00387_gb300 as kd
    kd.load()
    torch.cuda.init()
    return kd


def step(kd, flow, n, b, nsteps=2, limit=0):
    """(states, device bytes held)"""
    import torch
    ctx = kd.kd_create(kd.make_params(flow, n, 0.57, 50.0, 0.32 / n, kd.KD_C128))
    try:
        kd.kd_set_alloc_limit(ctx, limit)
        x = torch.tensor(b, dtype=torch.complex128, device="cuda")
        y = torch.full_like(x, float("nan"))
        t0 = 0.2 + 0.7 * torch.arange(len(b), dtype=torch.float64, device="cuda")
        kd.kd_fine_batched(ctx, x, y, t0, nsteps, len(b), kd.KD_C128)
        torch.cuda.synchronize()
        return y.cpu().numpy(), kd.kd_get_alloc_bytes(ctx)[0]
    finally:
        kd.kd_destroy(ctx)


# 192: the smallest kept set; 194 and 238 have 160 columns in the shared workspace, which the launches' 192
# exceed; 286: the largest set.  24 fields by launches, 25 in clusters
@pytest.mark.parametrize("flow", [O.ROBERTS, O.GALLOWAY_PROCTOR])
@pytest.mark.parametrize("n", [192, 194, 238, 286])
def test_launches_and_clusters_give_the_same_bits(kd, n, flow):
    b = I.initial_batch(n, 0.57, range(5))
    many = step(kd, flow, n, np.tile(b, (5, 1, 1, 1)))[0]
    for fields in (1, 5, 24):
        assert np.array_equal(step(kd, flow, n, np.tile(b, (5, 1, 1, 1))[:fields])[0], many[:fields]), fields


def test_without_room_for_the_launches(kd):
    """An allocation limit that holds the workspace of 160 columns but not of 192."""
    n = 200
    b = I.initial_batch(n, 0.57, [1])
    full, held = step(kd, O.GALLOWAY_PROCTOR, n, b)
    wider = 3 * (2 * (n // 3) + 1) * (192 - 160) * 16
    less, held2 = step(kd, O.GALLOWAY_PROCTOR, n, b, limit=held - wider)
    assert held2 == held - wider and np.array_equal(less, full)
    with pytest.raises(kd.KdError):
        step(kd, O.GALLOWAY_PROCTOR, n, b, limit=held - wider - 256)


# 16 (K = 5) and 22 (K = 7): two fields' rows share a warp, odd numbers of rows; 24 (K = 8): 32 points
@pytest.mark.parametrize("n", [16, 18, 22, 24])
@pytest.mark.parametrize("fields", [1, 3, 200])
def test_sixteen_points(kd, n, fields):
    b = np.stack([I.flat_field(n, 0.57, i) for i in range(min(fields, 3))])
    x = np.concatenate([b] * (-(-fields // len(b))))[:fields]
    for flow in (O.ROBERTS, O.GALLOWAY_PROCTOR):
        y = step(kd, flow, n, x, 3)[0]
        p = O.Problem(flow, n, 0.57, 50.0)
        for i in {0, len(b) - 1, fields - 1}:
            ref = O.propagate(x[i], p, 0.2 + 0.7 * i, 0.32 / n, 3)
            # ~30 rounded operations a stage, 12 stages: 360 unit roundoffs at the very most
            assert np.linalg.norm(y[i] - ref) < 4e-14 * np.linalg.norm(ref), i

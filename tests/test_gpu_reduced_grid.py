"""The complex64 RK443 step evaluated on the smallest suitable grid (3n/4 points for a
power-of-two side n: the flows hold only the wavenumbers +-1, so u x b of the kept modes has
no aliasing there) against the n-point kernels (launch plan (0, 0)) and the oracle.

Tolerances: both sides are complex64 steps of the same discrete operator, so they differ by
FP32 round-off of a few transforms a stage, about 2e-7 relative a step as every other launch
plan does (1e-6 bound, as in test_every_launch_plan_matches_oracle); 1e-5 against the oracle."""
import numpy as np
import pytest

import kd_inputs as I
from oracle import kd_oracle as O

pytestmark = pytest.mark.gpu

NO_FLOW = 2


@pytest.fixture(scope="module")
def kd():
    import torch
    import __graft_entry__
    __graft_entry__.build()
    import paper_1902_00387_gb300 as kd
    kd.load()
    torch.cuda.init()
    return kd


def rel(a, b):
    return float(np.linalg.norm((a - b).ravel()) / np.linalg.norm(b.ravel()))


def kept(b):
    n = b.shape[-1]
    i = np.arange(-(n // 3), n // 3 + 1) % n
    return np.ascontiguousarray(b[..., i, :][..., i])


def step(kd, flow, n, b, t0, nsteps, plan, layout):
    import torch
    ctx = kd.kd_create(kd.make_params(flow, n, 0.57, 1e3, 0.64 / n, kd.KD_C64))
    try:
        if plan is not None:
            kd.kd_set_plan(ctx, kd.KD_GRID_FINE, *plan)
        x = torch.tensor(kept(b) if layout == "kept" else b, dtype=torch.complex64, device="cuda")
        y = torch.full_like(x, float("nan"))
        call = kd.kd_fine_batched_kept if layout == "kept" else kd.kd_fine_batched
        call(ctx, x, y, torch.tensor(t0, dtype=torch.float64, device="cuda"), nsteps, len(t0))
        torch.cuda.synchronize()
        return y.cpu().numpy().astype(np.complex128)
    finally:
        kd.kd_destroy(ctx)


# 512: a block of the row kernel takes two of the 341 ky rows of a field, so odd batches end
# in half a block and even ones have blocks that straddle two fields; 1024: one row a block
@pytest.mark.parametrize("layout", ["full", "kept"])
@pytest.mark.parametrize("flow", [O.ROBERTS, O.GALLOWAY_PROCTOR, NO_FLOW])
@pytest.mark.parametrize("n,batch,nsteps", [(512, 1, 2), (512, 2, 1), (512, 3, 3), (1024, 1, 2), (1024, 2, 1)])
def test_default_plan_equals_the_n_point_kernels(kd, n, batch, nsteps, flow, layout):
    b = np.stack([I.flat_field(n, 0.57, 7 + i) for i in range(batch)])
    t0 = [0.3 + 1.7 * i for i in range(batch)]
    ref = step(kd, flow, n, b, t0, nsteps, (0, 0), layout)
    out = step(kd, flow, n, b, t0, nsteps, None, layout)
    for i in range(batch):
        assert rel(out[i], ref[i]) < 1e-6, i


def test_512_matches_oracle(kd):
    n = 512
    b = I.initial_batch(n, 0.57, [3, 4, 5])
    t0 = [0.0, 1.3, 7.9]
    out = step(kd, O.GALLOWAY_PROCTOR, n, b, t0, 4, None, "full")
    p = O.Problem(O.GALLOWAY_PROCTOR, n, 0.57, 1e3)
    for i in range(3):
        assert rel(out[i], O.propagate(b[i], p, t0[i], 0.64 / n, 4)) < 1e-5, i

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
@pytest.mark.parametrize("n,batch,nsteps", [(512, 4, 2), (512, 5, 1), (512, 7, 3), (1024, 1, 2), (1024, 2, 1)])
def test_default_plan_equals_the_n_point_kernels(kd, n, batch, nsteps, flow, layout):
    b = np.stack([I.flat_field(n, 0.57, 7 + i) for i in range(batch)])
    t0 = [0.3 + 1.7 * i for i in range(batch)]
    ref = step(kd, flow, n, b, t0, nsteps, (0, 0), layout)
    out = step(kd, flow, n, b, t0, nsteps, None, layout)
    for i in range(batch):
        assert rel(out[i], ref[i]) < 1e-6, i


def test_512_matches_oracle(kd):
    n = 512
    b = I.initial_batch(n, 0.57, [3, 4, 5, 6])
    t0 = [0.0, 1.3, 7.9, 2.2]
    out = step(kd, O.GALLOWAY_PROCTOR, n, b, t0, 4, None, "full")
    p = O.Problem(O.GALLOWAY_PROCTOR, n, 0.57, 1e3)
    for i in range(4):
        assert rel(out[i], O.propagate(b[i], p, t0[i], 0.64 / n, 4)) < 1e-5, i


# The persistent fused step: sides at the edges of its transform lengths (kept sets K = 5, 10 | 11,
# 23 | 24, 47 | 48, 63 | 64, 85, 95 for 24 (32 in complex128), 48, 96, 128, 192 points; K = 11, 12
# are n = 34, 36 and so on), batches of one field and of several.
FUSED_SIDES = [16, 32, 34, 36, 64, 70, 72, 128, 142, 144, 190, 192, 256, 286]


@pytest.mark.parametrize("n", FUSED_SIDES)
@pytest.mark.parametrize("prec", ["c64", "c128"])
def test_fused_step_matches_oracle(kd, n, prec):
    """Two steps of three fields (seven at n = 256, where fewer take the 256-point kernels) against the oracle's n-point steps, both flows; one field alone
    gives the same values bit for bit (the batch only decides how many blocks share a field)."""
    import torch
    pf = kd.KD_C64 if prec == "c64" else kd.KD_C128
    dtype = torch.complex64 if prec == "c64" else torch.complex128
    for flow in (O.ROBERTS, O.GALLOWAY_PROCTOR):
        nf = 7 if n == 256 else 3
        b = np.stack([I.flat_field(n, 0.57, 20 + i) for i in range(nf)])
        t0 = 0.2 + 1.7 * np.arange(nf)
        ctx = kd.kd_create(kd.make_params(flow, n, 0.57, 50.0, 0.32 / n, pf))
        try:
            x = torch.tensor(b, dtype=dtype, device="cuda")
            y, z = torch.full_like(x, float("nan")), torch.full_like(x[:1], float("nan"))
            tt = torch.tensor(t0, device="cuda")
            kd.kd_fine_batched(ctx, x, y, tt, 2, nf, pf)
            kd.kd_fine_batched(ctx, x[1:2].contiguous(), z, tt[1:2].contiguous(), 2, 1, pf)
            torch.cuda.synchronize()
        finally:
            kd.kd_destroy(ctx)
        assert n == 256 or torch.equal(y[1], z[0])
        p = O.Problem(flow, n, 0.57, 50.0)
        for i in (0, 2):
            ref = O.propagate(b[i], p, t0[i], 0.32 / n, 2)
            assert rel(y[i].cpu().numpy().astype(np.complex128), ref) < (1e-5 if prec == "c64" else 1e-12), i


@pytest.mark.parametrize("n,batch", [(64, 301), (128, 98), (192, 42), (256, 28)])
def test_fused_step_in_several_waves(kd, n, batch):
    """More fields than run at once, in one cluster shape, against seven of them in another."""
    import torch
    base = torch.tensor(I.initial_batch(n, 0.57, range(7)), dtype=torch.complex64, device="cuda")
    x = base.repeat(batch // 7, 1, 1, 1)
    t0 = torch.arange(batch, dtype=torch.float64, device="cuda") % 7
    ctx = kd.kd_create(kd.make_params(O.GALLOWAY_PROCTOR, n, 0.57, 100.0, 0.64 / n, kd.KD_C64))
    try:
        y, z = torch.empty_like(x), torch.empty_like(base)
        kd.kd_fine_batched(ctx, x, y, t0, 7, batch)
        kd.kd_fine_batched(ctx, base, z, t0[:7].contiguous(), 7, 7)
        torch.cuda.synchronize()
    finally:
        kd.kd_destroy(ctx)
    assert torch.equal(y, z.repeat(batch // 7, 1, 1, 1))


@pytest.mark.parametrize("n,batch,chunk", [(256, 8, 3), (512, 4, 2), (512, 3, 1)])
def test_chunks_take_the_plan_of_the_whole_call(kd, n, batch, chunk):
    """A host-buffer call in chunks below the few-field limit steps as the whole batch does."""
    import torch
    b = torch.tensor(I.initial_batch(n, 0.57, range(batch)), dtype=torch.complex64)
    t0 = np.arange(batch, dtype=np.float64)
    ctx = kd.kd_create(kd.make_params(O.GALLOWAY_PROCTOR, n, 0.57, 1e3, 0.64 / n, kd.KD_C64))
    try:
        h, d = torch.empty_like(b), torch.empty_like(b, device="cuda")
        kd.kd_fine_batched_host(ctx, b, h, t0, 2, batch, chunk)
        kd.kd_fine_batched(ctx, b.cuda(), d, torch.tensor(t0, device="cuda"), 2, batch)
        torch.cuda.synchronize()
    finally:
        kd.kd_destroy(ctx)
    assert torch.equal(h, d.cpu())

"""Parareal sweeps, batched sweeps and training pairs step with the plan of as many fields as the
whole call has (few or many: at 256^2 and 512^2 in complex64 these differ): the bits of
kd_fine_batched on as many fields."""
import numpy as np
import pytest

import kd_inputs as I
from oracle import kd_oracle as O

pytestmark = pytest.mark.gpu

DT = 2.0 ** -9       # slices of two steps whose lengths divide exactly
S = 2


@pytest.fixture(scope="module")
def kd():
    import torch
    import __graft_entry__
    __graft_entry__.build()
    import paper_1902_00387_gb300 as kd
    kd.load()
    torch.cuda.init()
    return kd


def context(kd, n, **more):
    return kd.kd_create(kd.make_params(O.GALLOWAY_PROCTOR, n, 0.57, 1e3, DT, kd.KD_C64, n_coarse=64, dt_coarse=DT,
                                       **more))


def batched(kd, n, b, t0):
    import torch
    ctx = context(kd, n)
    try:
        x = torch.as_tensor(b).to("cuda", torch.complex64)
        y = torch.empty_like(x)
        kd.kd_fine_batched(ctx, x, y, torch.tensor(t0, dtype=torch.float64, device="cuda"), S, len(b))
        torch.cuda.synchronize()
        return y.cpu().numpy()
    finally:
        kd.kd_destroy(ctx)


@pytest.mark.parametrize("form", ["direct", "increment"])
@pytest.mark.parametrize("n,slices", [(256, 1), (256, 3), (256, 4), (512, 2), (512, 3)])
def test_parareal_slices(kd, n, slices, form):
    """After one iteration the first slice's end is F(b0)."""
    b0 = I.initial_field(n, 0.57, 3)
    ctx = context(kd, n, fine_form=kd.KD_FINE_INCREMENT if form == "increment" else kd.KD_FINE_DIRECT)
    try:
        u = np.zeros((slices + 1, 3, n, n), np.complex128)
        kd.kd_parareal_run(ctx, b0, slices * S * DT, slices, 1, 0.0, u)
    finally:
        kd.kd_destroy(ctx)
    ref = batched(kd, n, np.repeat(b0[None], slices, 0), [0.0] * slices)[0]
    assert np.array_equal(u[1], ref.astype(np.complex128))


@pytest.mark.parametrize("instances", [1, 3, 4])
def test_sweep_of_single_slices(kd, instances):
    n = 256
    b = [I.initial_field(n, 0.57, i) for i in range(instances)]
    u = [np.zeros_like(x) for x in b]
    sw = kd.kd_sweep_create([kd.make_instance(O.GALLOWAY_PROCTOR, n, 0.57, 1e3, DT, 64, DT)] * instances, S * DT, 1)
    try:
        kd.kd_sweep_exec(sw, b, 1, 0.0, u_final=u)
    finally:
        sw.close()
    ref = batched(kd, n, np.stack(b), [0.0] * instances)
    for i in range(instances):
        assert np.array_equal(u[i], ref[i].astype(np.complex128)), i


@pytest.mark.parametrize("pairs", [2, 4])
def test_training_pairs(kd, pairs):
    import torch
    n, m = 256, 9
    k = np.arange(-(m // 2), m // 2 + 1) % n
    b = np.zeros((pairs, 3, n, n), np.complex64)
    x = np.ascontiguousarray(I.initial_batch(n, 0.57, range(pairs))[:, :, k][:, :, :, k].astype(np.complex64))
    b[:, :, k[:, None], k[None, :]] = x
    ctx = context(kd, n, learned_modes=m, fine_form=kd.KD_FINE_INCREMENT)
    try:
        kd.kd_learned_init(ctx, 1, S * DT)
        y = torch.empty((pairs, 3, m, m), dtype=torch.complex64, device="cuda")
        kd.kd_learned_pairs(ctx, torch.tensor(x, device="cuda"), pairs, [0] * pairs, y)
    finally:
        kd.kd_destroy(ctx)
    ref = batched(kd, n, b, [0.0] * pairs)[:, :, k][:, :, :, k]
    assert np.array_equal(y.cpu().numpy(), ref)


# fields and the largest chunk without a lower bound on chunks
@pytest.mark.parametrize("n,fields,largest", [(256, 5, 1), (256, 16, 4), (512, 3, 1), (512, 9, 2)])
def test_graded_chunks_of_host_fields(kd, n, fields, largest):
    """Chunks of a host-buffer call that are larger than a few fields: the device call's bits, also in
    place and under an allocation limit that has room for the smaller chunks only."""
    import torch
    b = torch.tensor(I.initial_batch(n, 0.57, range(fields)), dtype=torch.complex64)
    t0 = np.arange(fields, dtype=np.float64)
    ref = batched(kd, n, b, t0)
    limit = 0
    for chunk in (largest, 0, 0):
        ctx = context(kd, n)
        try:
            kd.kd_set_alloc_limit(ctx, limit)
            y = b.clone()
            kd.kd_fine_batched_host(ctx, y, y, t0, S, fields, chunk)
            assert np.array_equal(y.numpy(), ref)
            held = kd.kd_get_alloc_bytes(ctx)[0]
            assert not limit or held <= limit
            limit = 0 if chunk == 0 else held
        finally:
            kd.kd_destroy(ctx)

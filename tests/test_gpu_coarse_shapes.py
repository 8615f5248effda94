"""The cluster sizes that the coarse solver takes for a batch: a field's values are the same bits
in every batch, those of one field alone, and the oracle's."""
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


def conv_fine(kd, n, prec, b, t0, nsteps, cluster=0):
    import torch
    ctx = kd.kd_create(kd.make_params(O.GALLOWAY_PROCTOR, n, 0.57, 100.0, 5e-3, prec, fine_operator=kd.KD_FINE_CONV))
    try:
        if cluster:
            kd.kd_set_coarse_cluster(ctx, cluster)
        x = torch.tensor(b, dtype=torch.complex64 if prec == kd.KD_C64 else torch.complex128, device="cuda")
        y = torch.empty_like(x)
        kd.kd_fine_batched(ctx, x, y, torch.tensor(t0, dtype=torch.float64, device="cuda"), nsteps, len(b), prec)
        torch.cuda.synchronize()
        return y.cpu().numpy()
    finally:
        kd.kd_destroy(ctx)


# one block a field (n = 16), one wave, several waves; rows that divide unevenly (n = 64, 100);
# 128: 85 rows in 15 blocks alone, 10 or so of 9 rows in a batch (two modes a thread, 16 warps)
@pytest.mark.parametrize("n,fields", [(16, 200), (32, 64), (64, 7), (64, 64), (100, 16), (128, 20), (128, 64)])
@pytest.mark.parametrize("prec", ["c64", "c128"])
def test_batch_equals_single_field(kd, n, fields, prec):
    if prec == "c128" and fields > 20:
        fields = 20
    P = kd.KD_C64 if prec == "c64" else kd.KD_C128
    b = I.initial_batch(n, 0.57, [91 + i for i in range(fields)])
    t0 = [0.3 * i for i in range(fields)]
    out = conv_fine(kd, n, P, b, t0, 3)
    p = O.Problem(O.GALLOWAY_PROCTOR, n, 0.57, 100.0)
    for i in {0, fields // 2, fields - 1}:
        assert np.array_equal(out[i], conv_fine(kd, n, P, b[i:i + 1], t0[i:i + 1], 3)[0])
    ref = O.propagate(b[-1], p, t0[-1], 5e-3, 3)
    # ~30 rounded operations a stage, 12 stages: 360 unit roundoffs at the very most
    assert np.linalg.norm(out[-1] - ref) < (2.2e-5 if prec == "c64" else 4e-14) * np.linalg.norm(ref)


@pytest.mark.parametrize("cluster", [8, 9, 11, 13, 16])
def test_two_modes_a_thread_at_every_fill(kd, cluster):
    """513 to 1024 modes a block (9: 850, 8: 935 of 1024 slots), beside one mode a thread (16)."""
    b = I.initial_batch(128, 0.57, [91, 92])
    one = conv_fine(kd, 128, kd.KD_C64, b, [0.0, 0.7], 4)
    assert np.array_equal(conv_fine(kd, 128, kd.KD_C64, b, [0.0, 0.7], 4, cluster), one)

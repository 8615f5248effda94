"""|W - W0|^2 of the learned objective, which the loss returns in double: as precise as an FP64 sum."""
from fractions import Fraction

import numpy as np
import pytest

from oracle import kd_oracle as O

pytestmark = pytest.mark.gpu


# differences that are no FP32 numbers, without and with several elements a thread (m = 32: 72);
# equal elements, so that no rounding averages out
@pytest.mark.parametrize("m", [5, 32])
@pytest.mark.parametrize("w,w0", [(-0.5356694, 0.00036159504), (-1.245911, -0.00073226733), (0.64042264, 1.04900115e-4)])
def test_norm_has_fp64_precision(m, w, w0):
    """The squares' sum is exact but for the additions across threads: 5 in a warp, 8 in a block, the
    blocks' sums in at most 4 + 8 + 5 steps and the result's own roundings, fewer than 40 of 2^-53."""
    import torch
    import __graft_entry__
    __graft_entry__.build()
    import paper_1902_00387_gb300 as kd
    nc = 3 * m * m
    W = torch.full((2 * nc, nc), w, dtype=torch.float32, device="cuda")
    W0 = torch.full_like(W, w0)
    x = torch.zeros((4, nc), dtype=torch.complex64, device="cuda")
    ctx = kd.kd_create(kd.make_params(O.ROBERTS, 128, 0.57, 100.0, 0.01, kd.KD_C64, n_coarse=64, dt_coarse=0.04,
                                      prec_coarse=kd.KD_C64, learned_modes=m))
    try:
        loss = kd.kd_learned_loss_grad(ctx, W, W0, 1.0, x, x, 4, torch.empty_like(W))
    finally:
        kd.kd_destroy(ctx)
    exact = 2 * nc * nc * (Fraction(float(np.float32(w))) - Fraction(float(np.float32(w0)))) ** 2
    assert abs(Fraction(loss) / exact - 1) < 40 * Fraction(1, 2 ** 53)

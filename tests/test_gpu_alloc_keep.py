"""Training buffers that a context keeps between calls: reused by a call of the same size, given
back before an allocation limit refuses anything, and the same values either way."""
import numpy as np
import pytest

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


def test_buffers_are_reused_and_given_back(kd):
    import torch
    P, nc = 8, 192
    rng = np.random.default_rng(3)
    W = torch.tensor(0.1 * rng.standard_normal((2 * nc, nc)), dtype=torch.float32, device="cuda")
    X = torch.tensor(rng.standard_normal((64, nc, 2)), dtype=torch.float32, device="cuda")
    X = torch.view_as_complex(X)
    ctx = kd.kd_create(kd.make_params(O.ROBERTS, 32, 0.57, 8.0, 0.01, kd.KD_C64, n_coarse=16, dt_coarse=0.04,
                                      prec_coarse=kd.KD_C64, learned_modes=P))
    try:
        def grad(m):
            g = torch.empty((2 * nc, nc), dtype=torch.float32, device="cuda")
            return kd.kd_learned_loss_grad(ctx, W, None, 0.1, X[:m], X[:m], m, g), g.cpu().numpy()

        held0 = kd.kd_get_alloc_bytes(ctx)[0]
        l64, g64 = grad(64)
        held1 = kd.kd_get_alloc_bytes(ctx)[0]
        assert held1 > held0
        l5, g5 = grad(5)
        grad(64)
        held2 = kd.kd_get_alloc_bytes(ctx)[0]
        for m, l, g in ((64, l64, g64), (5, l5, g5)):      # both sizes from kept buffers
            l2, g2 = grad(m)
            assert l2 == l and np.array_equal(g2, g)
            assert kd.kd_get_alloc_bytes(ctx)[0] == held2
        # a limit that refused the call before it kept anything refuses it still
        kd.kd_set_alloc_limit(ctx, held0 + 1000)
        with pytest.raises(RuntimeError, match="allocation limit"):
            grad(64)
        kd.kd_set_alloc_limit(ctx, held1)
        kd.kd_set_alloc_limit(ctx, 0)
        l2, g2 = grad(64)
        assert l2 == l64 and np.array_equal(g2, g64)
        # kept buffers of another size make room for a call that fits the limit without them
        used = kd.kd_get_alloc_bytes(ctx)[0]
        kd.kd_set_alloc_limit(ctx, used)
        l2, g2 = grad(60)
        assert kd.kd_get_alloc_bytes(ctx)[0] <= used
        assert abs(l2 - grad(60)[0]) == 0
    finally:
        kd.kd_destroy(ctx)

"""Gradient and norm pass of the learned training objective at the edges of its tiles: odd and
even numbers of unknowns, one pair to several tiles of them, with and without a centre W0."""
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


def loss_grad(kd, P, W, W0, wd, X, Y):
    import torch
    ctx = kd.kd_create(kd.make_params(O.ROBERTS, 32, 0.57, 8.0, 0.01, kd.KD_C64, n_coarse=16, dt_coarse=0.04,
                                      prec_coarse=kd.KD_C64, learned_modes=P))
    try:
        nc = 3 * P * P
        g = torch.full((2 * nc, nc), np.nan, dtype=torch.float32, device="cuda")
        t = [None if a is None else torch.tensor(a, device="cuda") for a in (W, W0, X, Y)]
        loss = kd.kd_learned_loss_grad(ctx, t[0], t[1], wd, t[2], t[3], len(X), g)
        return loss, g.cpu().numpy().astype(np.float64)
    finally:
        kd.kd_destroy(ctx)


@pytest.mark.parametrize("P,m,centre", [(3, 1, True), (5, 5, False), (6, 32, True), (7, 33, False), (11, 70, True)])
def test_gradient_at_tile_edges(kd, P, m, centre):
    rng = np.random.default_rng(P)
    nc, wd = 3 * P * P, 0.05
    W = (0.1 * rng.standard_normal((2 * nc, nc))).astype(np.float32)
    W0 = (0.1 * rng.standard_normal((2 * nc, nc))).astype(np.float32) if centre else None
    X, Y = ((rng.standard_normal((m, nc)) + 1j * rng.standard_normal((m, nc))).astype(np.complex64) for _ in range(2))
    loss, g = loss_grad(kd, P, W, W0, wd, X, Y)
    Wc = W[:nc].astype(np.float64) + 1j * W[nc:]
    W0c = 0 * Wc if W0 is None else W0[:nc].astype(np.float64) + 1j * W0[nc:]
    ex_loss, ex = O.learned_loss_grad(Wc, X.astype(np.complex128), Y.astype(np.complex128), W0c, wd)
    # BF16 operands: W, X and the residual are rounded once each, 2^-9 a factor, independently
    # over the sums; 2 % is 10 of these roundings
    assert abs(loss - ex_loss) < 2e-2 * ex_loss
    assert np.linalg.norm(g[:nc] + 1j * g[nc:] - ex) < 2e-2 * np.linalg.norm(ex)


@pytest.mark.parametrize("P,scale", [(4, 1.0), (5, 1e-18), (9, 1e18), (10, 1e-2)])
def test_decay_term_alone(kd, P, scale):
    """Without data the gradient is 2 wd (W - W0), rounded twice, and the loss its norm, in which
    squares beyond FP32's range have their own sum."""
    rng = np.random.default_rng(100 + P)
    nc, wd = 3 * P * P, 0.25
    spread = 10.0 ** rng.uniform(-3, 3, (2 * nc, nc))
    W = (scale * spread * rng.standard_normal((2 * nc, nc))).astype(np.float32)
    W0 = (W * (1 + 1e-3 * rng.standard_normal(W.shape))).astype(np.float32)
    W0[::3] = W[::3]
    zero = np.zeros((6, nc), np.complex64)
    loss, g = loss_grad(kd, P, W, W0, wd, zero, zero)
    d = W.astype(np.float64) - W0
    assert np.max(np.abs(g - 2 * wd * d) - 2.0 ** -22 * np.abs(2 * wd * d)) <= 0
    # a thread's pair of floats keeps each addition to about 2^-46 of the sum
    assert abs(loss - wd * np.sum(d * d)) < 1e-11 * wd * np.sum(d * d)

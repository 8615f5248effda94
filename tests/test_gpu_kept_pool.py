"""Training buffers that contexts keep between calls: each its own, given back when another context finds
the GPU full."""
import pytest

from oracle import kd_oracle as O

pytestmark = pytest.mark.gpu

M = 49                       # 0.62 GB of buffers


@pytest.fixture(scope="module")
def kd():
    import torch
    import __graft_entry__
    __graft_entry__.build()
    import paper_1902_00387_gb300 as kd
    kd.load()
    torch.cuda.init()
    return kd


def context(kd):
    return kd.kd_create(kd.make_params(O.ROBERTS, 256, 0.57, 100.0, 0.01, kd.KD_C64, n_coarse=64, dt_coarse=0.04,
                                       learned_modes=M))


def held(kd, ctx):
    return kd.kd_get_alloc_bytes(ctx)[0]


@pytest.fixture
def objective(kd):
    import torch
    nc = 3 * M * M
    W = torch.zeros((2 * nc, nc), device="cuda")
    x = torch.randn((64, nc), dtype=torch.complex64, device="cuda")
    g = torch.empty_like(W)
    return lambda ctx: kd.kd_learned_loss_grad(ctx, W, None, 0.0, x, x, 64, g)


def test_contexts_keep_their_own(kd, objective):
    """Two contexts in turn: each holds the same bytes after every call, and the end of one leaves the
    other's alone."""
    a, b = context(kd), context(kd)
    try:
        free = held(kd, a)
        la, lb = objective(a), objective(b)
        kept = held(kd, a) - free
        assert 5e8 < kept <= 2 ** 30 and held(kd, b) - free == kept
        assert objective(a) == la == lb and objective(b) == lb
        assert held(kd, a) - free == held(kd, b) - free == kept
    finally:
        kd.kd_destroy(a)
    try:
        assert held(kd, b) - free == kept and objective(b) == lb
    finally:
        kd.kd_destroy(b)


def test_a_full_gpu_takes_them_back_for_any_context(kd, objective):
    import torch
    a, b = context(kd), context(kd)
    fill = None
    try:
        before = held(kd, a)
        objective(a)
        kept = held(kd, a) - before
        assert kept > 5e8
        x = torch.zeros((32, 3, 256, 256), dtype=torch.complex64, device="cuda")
        y, t0 = torch.empty_like(x), torch.zeros(32, dtype=torch.float64, device="cuda")
        torch.cuda.empty_cache()
        # leave less than the call's workspace (180 MB), which the kept buffers make room for
        fill = torch.empty(torch.cuda.mem_get_info()[0] - 2 ** 27, dtype=torch.uint8, device="cuda")
        kd.kd_fine_batched(b, x, y, t0, 1, 32)
        torch.cuda.synchronize()
        assert held(kd, a) == before and float(y.abs().max()) == 0.0
    finally:
        del fill
        torch.cuda.empty_cache()
        kd.kd_destroy(a)
        kd.kd_destroy(b)

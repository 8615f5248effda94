"""Rounding error of the complex64 defaults, which step on 3n/4 points, against 64 bits and against that
of the n-point kernels (plan (0, 0))."""
import numpy as np
import pytest

import kd_inputs as I
from oracle import kd_oracle as O

pytestmark = pytest.mark.gpu


# batches that take the default of many fields
@pytest.mark.parametrize("n,fields,nsteps", [(64, 6, 20), (128, 6, 10), (256, 7, 3), (512, 3, 2), (1024, 1, 1)])
def test_three_quarters_of_the_points(n, fields, nsteps):
    """White noise on N points leaves P^2 / N^2 of its variance in the kept modes, so the amplitude grows
    by n / N = 4/3 at most, less where the error is the state's own; a tenth for the other radices."""
    import torch
    import __graft_entry__
    __graft_entry__.build()
    import paper_1902_00387_gb300 as kd
    kz, Rm, dt = 0.57, 8.0 * (n / 32.0) ** 2, 0.64 / n
    b = I.initial_batch(n, kz, range(40, 40 + fields)).astype(np.complex64)
    p = O.Problem(O.GALLOWAY_PROCTOR, n, kz, Rm)
    ref = O.propagate(b[0].astype(np.complex128), p, 0.3, dt, nsteps)

    def error(plan):
        ctx = kd.kd_create(kd.make_params(O.GALLOWAY_PROCTOR, n, kz, Rm, dt, kd.KD_C64))
        try:
            if plan:
                kd.kd_set_plan(ctx, kd.KD_GRID_FINE, *plan)
            x = torch.tensor(b, device="cuda")
            y = torch.empty_like(x)
            kd.kd_fine_batched(ctx, x, y, torch.full((fields,), 0.3, dtype=torch.float64, device="cuda"), nsteps, fields)
            return np.linalg.norm(y[0].cpu().numpy() - ref)
        finally:
            kd.kd_destroy(ctx)

    assert error(None) < 1.1 * 4 / 3 * error((0, 0))

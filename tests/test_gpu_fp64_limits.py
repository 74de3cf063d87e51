"""FP64 digit products (kernel 11 on FP64 values, kernel 10 on those of 9 x 9 systems) at the limits of their
operands: NaN and infinities met while the operands are split, results at the ends of the exponent range."""
import numpy as np
import pytest
import torch

from paper_0911_3584_gb300 import Context, Pattern, Plan
from tests.gpu_util import to_dev

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx(cuda_device):
    return Context(cuda_device)


@pytest.mark.parametrize("row", [0, 1, 700])
def test_nan_in_one_row_of_thousands(ctx, row):
    """A NaN that one CTA of the splitting kernel meets while the others start: the blocks of every row but the
    NaN's come out as without it, whichever CTAs know of it, call after call."""
    rng = np.random.default_rng(row)
    n = 5000
    pos, cell = rng.uniform(0, 60.0, size=(n, 3)), np.array([60.0, 60.0, 60.0])
    P = Pattern.build(ctx, pos, cell, 5.0)
    rp = P.row_ptr.cpu().numpy()
    a, b = (rng.standard_normal((P.nnzb, 4, 4)) for _ in "ab")
    a[rp[row], 1, 2] = np.nan
    ref_plan, plan = Plan(ctx, P, P, P, trans_b=True), Plan(ctx, P, P, P, trans_b=True)
    ref_plan.set_kernel("triples")
    plan.set_kernel("tensor-tile")
    dev = [to_dev(v, torch.float64, ctx.device) for v in (a, b)]
    ref = ref_plan.multiply(*dev)
    fine = torch.isfinite(ref)
    assert not fine.all() and fine[rp[row + 1]:].all()
    for _ in range(20):
        C = plan.multiply(*dev)
        assert torch.equal(torch.isnan(C), ~fine)
        assert (C[fine] - ref[fine]).norm() <= 1e-14 * ref[fine].norm()
    assert ctx.device_status() == 0

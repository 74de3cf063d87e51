"""FP64 digit products (kernel 11 on FP64 values, kernel 10 on those of 9 x 9 systems) at the limits of their
operands: NaN and infinities met while the operands are split, results at the ends of the exponent range."""
from fractions import Fraction

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


@pytest.mark.parametrize("a,b", [
    (1.5 * 2.0 ** 511, 2.0 ** 512),                      # 1.5 2^1023
    ((2.0 - 2.0 ** -52) * 2.0 ** 511, 2.0 ** 512),       # the largest finite value
    (2.0 ** 511, 2.0 ** 512),                            # 2^1023
    ((2.0 - 2.0 ** -52) * 2.0 ** 511, 2.0 ** 511),       # just below it
    (2.0 ** 512, 2.0 ** 512),                            # overflows
    (3 * 2.0 ** -500, 5 * 2.0 ** -520),                  # just above the smallest normal value
    (3 * 2.0 ** -530, 5 * 2.0 ** -543),                  # subnormal, exact
    (3 * 2.0 ** -538, 5 * 2.0 ** -538),                  # 15 / 4 units of 2^-1074
    (3 * 2.0 ** -540, 2.0 ** -538),                      # 3 / 16 units: rounds to zero
])
@pytest.mark.parametrize("sign", [1.0, -1.0])
def test_results_at_the_ends_of_the_exponent_range(ctx, a, b, sign):
    """One term per element: its correctly rounded value, in every row and column of a block."""
    P = Pattern.build(ctx, np.zeros((1, 3)) + 1.0, np.array([50.0, 50.0, 50.0]), 3.0)
    A, B = np.zeros((1, 4, 4)), np.zeros((1, 4, 4))
    A[0, :, 1], B[0, 1, :] = sign * a, b
    exact = Fraction(a) * Fraction(b)
    want = sign * (float(exact) if exact < 2 ** 1024 - 2 ** 970 else np.inf)
    plan = Plan(ctx, P, P, P)
    plan.set_kernel("tensor-tile")
    C = plan.multiply(*(to_dev(v, torch.float64, ctx.device) for v in (A, B))).cpu().numpy()
    assert np.array_equal(C, np.full((1, 4, 4), want)), (C, want)


@pytest.mark.parametrize("k", [4, 9, 20, 33])
def test_subnormal_results_are_rounded_once(ctx, k):
    """A product of 54 bits whose last k bits, just below one half, are lost: a rounding to 53 bits on the way makes
    them one half, and a second one rounds that up."""
    p = 2 ** 53 + 2 ** (k - 1) - 1
    while p % 3:
        p += 2 ** k
    a, b = 3 * 2.0 ** -500, float(p // 3) * 2.0 ** (500 - 1074 - k)
    assert int(float(p // 3)) == p // 3
    P = Pattern.build(ctx, np.zeros((1, 3)) + 1.0, np.array([50.0, 50.0, 50.0]), 3.0)
    A, B = np.zeros((1, 4, 4)), np.zeros((1, 4, 4))
    A[0, :, 1], B[0, 1, :] = a, b
    plan = Plan(ctx, P, P, P)
    plan.set_kernel("tensor-tile")
    C = plan.multiply(*(to_dev(v, torch.float64, ctx.device) for v in (A, B))).cpu().numpy()
    want = float(Fraction(a) * Fraction(b))
    assert want == (p >> k) * 2.0 ** -1074
    assert np.array_equal(C, np.full((1, 4, 4), want)), (C / 2.0 ** -1074, p >> k)

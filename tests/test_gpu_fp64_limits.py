"""FP64 digit products (kernel 11 on FP64 values, kernel 10 on those of 9 x 9 systems) at the limits of their
operands: NaN and infinities met while the operands are split, results at the ends of the exponent range, buffers of
the digits that outlive a call."""
from fractions import Fraction

import numpy as np
import pytest
import torch

import oracle
from paper_0911_3584_gb300 import Context, Pattern, Plan, System
from tests.gpu_util import rel_fro, to_dev, workload

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


def _product(ctx, seed, n, cutoff):
    rng = np.random.default_rng(seed)
    P = Pattern.build(ctx, rng.uniform(0, 24.0, size=(n, 3)), np.array([24.0, 24.0, 24.0]), cutoff)
    plan = Plan(ctx, P, P, P, trans_b=True)
    plan.set_kernel("tensor-tile")
    return plan, [to_dev(rng.standard_normal((P.nnzb, 4, 4)), torch.float64, ctx.device) for _ in "ab"]


def _tuned_system(ctx):
    w, S, H, L = workload(2, 4, 6.6, 8.0, 7)
    sysm = System(ctx, 4, "fp64", w["pos"], w["cell"], 6.6, 8.0)
    sysm.autotune(*(to_dev(M["val"], torch.float64, ctx.device) for M in (S, H, L)), reps=1)


def test_captured_product_outlives_larger_ones(cuda_device):
    """A product captured in a graph replays with its bits after a larger product and an autotune on the same
    context, with other arrays allocated and filled in between; it needs no call before the capture."""
    ctx = Context(cuda_device)
    plan, (a, b) = _product(ctx, 1, 300, 5.0)
    C = torch.zeros((plan.C.nnzb, 4, 4), dtype=torch.float64, device=cuda_device)
    graph, side, old = torch.cuda.CUDAGraph(), torch.cuda.Stream(cuda_device), ctx.stream
    torch.cuda.synchronize()
    with torch.cuda.graph(graph, stream=side):
        ctx.set_stream(side)
        try:
            plan.multiply(a, b, C)
        finally:
            ctx.set_stream(old)
    want = plan.multiply(a, b)
    big, vals = _product(ctx, 2, 1200, 8.0)
    big.multiply(*vals)
    _tuned_system(ctx)
    torch.cuda.synchronize()
    junk = [torch.full((1 << 26,), float("nan"), dtype=torch.float64, device=cuda_device) for _ in range(4)]
    for _ in range(3):
        C.zero_()
        graph.replay()
        big.multiply(*vals)
        assert torch.equal(C, want)
    assert all(torch.isnan(j).all() for j in junk)
    assert ctx.device_status() == 0


def test_products_on_two_streams_of_one_context(cuda_device):
    """Products that take turns on two streams share no buffer."""
    ctx = Context(cuda_device)
    cases = [_product(ctx, k, n, 8.0) for k, n in enumerate((900, 700))]
    want = [plan.multiply(*v) for plan, v in cases]
    streams, old = [torch.cuda.Stream(cuda_device) for _ in cases], ctx.stream
    got = [[torch.empty_like(w) for _ in range(6)] for w in want]
    torch.cuda.synchronize()
    for i in range(6):
        for s, (plan, v), g in zip(streams, cases, got):
            ctx.set_stream(s)
            plan.multiply(*v, C_vals=g[i])
    ctx.set_stream(old)
    torch.cuda.synchronize()
    assert all(torch.equal(x, w) for g, w in zip(got, want) for x in g)
    assert ctx.device_status() == 0


@pytest.mark.parametrize("nsf", [4, 9])
def test_truncation_below_the_range_of_s(cuda_device, nsf):
    """r_t < r_sh: S has more blocks than T, whose place its digits do not fit; equal to the oracle, captured too, with
    an autotune of another system in between."""
    ctx = Context(cuda_device)
    from synth import si_diamond_positions, sym_block_values
    rng = np.random.default_rng(8)
    pos, cell = si_diamond_positions(2, rng)
    r_sh, r_l, r_x, r_t = 6.0, 3.0, 4.0, 4.0
    pat = {k: oracle.pattern(pos, cell, r) for k, r in (("S", r_sh), ("H", r_sh), ("L", r_l))}
    M = {k: oracle.csr(*pat[k], sym_block_values(*pat[k], pos, cell, nsf, k, rng)) for k in "SHL"}
    ref = oracle.lnv_energy_grad_truncated(pos, cell, r_sh, r_l, r_x, r_t, M["S"], M["H"], M["L"])
    sysm = System(ctx, nsf, "fp64", pos, cell, r_sh, r_l, r_x=r_x, r_t=r_t)
    vals = [to_dev(M[k]["val"], torch.float64, ctx.device) for k in "SHL"]
    graph, out, G = sysm.capture(*vals)
    _tuned_system(ctx)
    for _ in range(2):
        out.zero_()
        G.zero_()
        graph.replay()
        assert abs(out[0, 0].item() - ref["E"]) <= 1e-12 * abs(ref["E"])
        assert abs(out[0, 1].item() - ref["Ne"]) <= 1e-12 * abs(ref["Ne"])
        assert rel_fro(G.cpu().numpy(), ref["G"]) <= 1e-13
    assert ctx.device_status() == 0

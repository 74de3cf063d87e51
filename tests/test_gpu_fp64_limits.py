"""FP64 digit products (kernel 11 on FP64 values, kernel 10 on those of 9 x 9 systems) at the limits of their
operands: NaN and infinities met while the operands are split, results at the ends of the exponent range, buffers of
the digits that outlive a call, operands whose elements differ by many powers of two."""
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


def _elementwise(ctx, n_atoms, a, b, ta, tb):
    """(|C - ref|, K |A||B|) of a product on the full pattern of n_atoms atoms, ref and |A||B| in long double."""
    n = n_atoms
    P = Pattern.build(ctx, np.random.default_rng(0).uniform(0, 5.0, size=(n, 3)), np.array([30.0, 30.0, 30.0]), 14.9)
    assert P.nnzb == n * n
    blocks = [np.ascontiguousarray(v.reshape(n, 4, n, 4).transpose(0, 2, 1, 3)).reshape(n * n, 4, 4) for v in
              (a.T if ta else a, b.T if tb else b)]
    plan = Plan(ctx, P, P, P, trans_a=ta, trans_b=tb)
    plan.set_kernel("tensor-tile")
    C = plan.multiply(*(to_dev(v, torch.float64, ctx.device) for v in blocks)).cpu().numpy()
    C = C.reshape(n, n, 4, 4).transpose(0, 2, 1, 3).reshape(4 * n, 4 * n)
    A, B = a.astype(np.longdouble), b.astype(np.longdouble)
    return np.abs(C - A @ B), 4 * n * (np.abs(A) @ np.abs(B))


@pytest.mark.parametrize("ta", [False, True])
@pytest.mark.parametrize("tb", [False, True])
@pytest.mark.parametrize("spread", [0, 5, 7, 20, 40, 60, 500])
def test_inner_index_of_any_scale(ctx, spread, ta, tb):
    """A D times D^-1 B with D of powers of two over a wide range: the bound K 2^-53 |A||B| of a plain FP64 sum, element
    by element.  The digits' bound is K 2^-53 max|row of A| max|column of B|, with the largest elements at most 2^4
    apart from those that they meet (the rest is formed term by term); 260 normal terms have |A||B| of about 166 and
    max max of at most 16, so that bound is below 2^4 16 / 166 < 2 times the plain sum's: 4 is allowed."""
    rng = np.random.default_rng(spread)
    d = 2.0 ** np.round(spread * rng.uniform(-0.5, 0.5, size=260))
    err, kab = _elementwise(ctx, 65, rng.standard_normal((260, 260)) * d, rng.standard_normal((260, 260)) / d[:, None],
                            ta, tb)
    assert np.all(err <= 4 * 2.0 ** -53 * kab), np.max(err / kab) / 2.0 ** -53


@pytest.mark.parametrize("tb", [False, True])
def test_large_element_that_meets_nothing(ctx, tb):
    """Rows whose largest element, by 2^60, multiplies a row of zeros of B; columns likewise: the rest is exact."""
    rng = np.random.default_rng(1)
    a, b = rng.standard_normal((2, 36, 36))
    a[:, 5] *= 2.0 ** 60
    b[5] = 0.0
    b[17] *= 2.0 ** 60
    a[:, 17] = 0.0
    err, kab = _elementwise(ctx, 9, a, b, False, tb)
    assert np.all(err <= 2.0 ** -53 * kab), np.max(err / kab) / 2.0 ** -53


def _rescaled(M, d, power):
    """Blocks ij of M times d_i^power on their rows and d_j^power on their columns (d [n, nsf])."""
    rows = np.repeat(np.arange(M["rp"].size - 1), np.diff(M["rp"]))
    return M["val"] * (d[rows] ** power)[:, :, None] * (d[M["col"]] ** power)[:, None, :]


@pytest.mark.parametrize("nsf", [4, 9])
@pytest.mark.parametrize("spread", [0, 4, 10, 20, 40, 60])
def test_evaluation_does_not_depend_on_the_scale_of_basis_functions(ctx, nsf, spread):
    """S -> D S D, H -> D H D, L -> D^-1 L D^-1 with powers of two: E, N_e and the traces stay, dE/dL becomes D G D."""
    rng = np.random.default_rng(spread)
    if nsf == 4:
        w, S, H, L = workload(2, 4, 6.6, 8.0, 5)
        pos, cell, r = w["pos"], w["cell"], (6.6, 8.0)
    else:
        from synth import si_diamond_positions, sym_block_values
        pos, cell = si_diamond_positions(2, rng)
        pos, r = np.ascontiguousarray(pos[:43]), (4.0, 6.0)
        pat = {k: oracle.pattern(pos, cell, c) for k, c in (("S", r[0]), ("H", r[0]), ("L", r[1]))}
        S, H, L = (oracle.csr(*pat[k], sym_block_values(*pat[k], pos, cell, 9, k, rng)) for k in "SHL")
    ref = oracle.lnv_energy_grad(pos, cell, *r, S, H, L, grad=True, grad_ne=True)
    d = 2.0 ** np.round(spread * rng.uniform(-0.5, 0.5, size=(pos.shape[0], nsf)))
    sysm = System(ctx, nsf, "fp64", pos, cell, *r)
    out, G, GN = sysm.energy_grad(*(to_dev(_rescaled(M, d, p), torch.float64, ctx.device) for M, p in
                                    ((S, 1.0), (H, 1.0), (L, -1.0))), grad_ne=True)
    back = [_rescaled(dict(L, val=g.cpu().numpy()), d, -1.0) for g in (G, GN)]
    assert abs(out[0, 0].item() - ref["E"]) <= 1e-12 * abs(ref["E"])
    assert abs(out[0, 1].item() - ref["Ne"]) <= 1e-12 * abs(ref["Ne"])
    assert rel_fro(back[0], ref["G"]) <= 1e-12
    assert rel_fro(back[1], ref["GN"]) <= 1e-12
    assert ctx.device_status() == 0


@pytest.mark.parametrize("bad", ["nan", "scale"])
@pytest.mark.parametrize("nsf", [4, 9])
def test_one_system_of_a_batch_does_not_touch_the_others(ctx, nsf, bad):
    """A NaN in one system, or one of badly scaled basis functions: the bits of the others stay (groups of atoms
    that the products take together span the systems)."""
    rng = np.random.default_rng(4)
    pos = [rng.uniform(0, 8.0, size=(n, 3)) for n in (21, 13, 18)]
    cell, off = [40.0, 40.0, 40.0], [0, 21, 34, 52]
    sysm = System(ctx, nsf, "fp64", np.concatenate(pos), [cell] * 3, 4.0, 5.0, seg_off=off)
    dev = ctx.device

    def vals(P, scale):
        rp, col, tr = P.row_ptr.cpu(), P.col.cpu().long(), P.tr.cpu()
        v = scale * torch.from_numpy(rng.standard_normal((P.nnzb, nsf, nsf)))
        v = 0.5 * (v + v[tr].transpose(1, 2))
        row = torch.repeat_interleave(torch.arange(P.n), rp[1:] - rp[:-1])
        v[row == col] += torch.eye(nsf, dtype=torch.float64)
        return v, row

    S, row = vals(sysm.P_sh, 0.05)
    H, _ = vals(sysm.P_sh, 0.3)
    L, _ = vals(sysm.P_l, 0.02)
    out0, G0 = sysm.energy_grad(S.to(dev), H.to(dev), L.to(dev))
    mid = (row >= 21) & (row < 34)
    if bad == "nan":
        H[int(mid.nonzero()[3]), 1, 2] = float("nan")
    else:
        d = 2.0 ** torch.from_numpy(np.round(30 * rng.uniform(size=(52, nsf))))
        S[mid] = (S * d[row][:, :, None] * d[sysm.P_sh.col.cpu().long()][:, None, :])[mid]
    out, G = sysm.energy_grad(S.to(dev), H.to(dev), L.to(dev))
    rp = sysm.P_l.row_ptr.cpu()
    keep = torch.cat([torch.arange(int(rp[21])), torch.arange(int(rp[34]), sysm.P_l.nnzb)]).to(dev)
    assert torch.equal(out[[0, 2]], out0[[0, 2]])
    assert torch.equal(G[keep], G0[keep])
    assert not torch.equal(out[1], out0[1])


@pytest.mark.parametrize("digits", ["XY", "TU", "Z", "Q", "W"])
@pytest.mark.parametrize("other", ["push", "pull", "group", "group-sparse", "triples"])
@pytest.mark.parametrize("mirror", [True, False])
def test_one_stage_on_digits_beside_plain_ones(ctx, digits, other, mirror):
    """U is formed after Z when T's digits take its place, on the kernel of T and U, and is not symmetric as T is."""
    w, S, H, L = workload(2, 4, 4.0, 5.0, 3)
    ref = oracle.lnv_energy_grad(w["pos"], w["cell"], 4.0, 5.0, S, H, L, grad=True, grad_ne=True)
    sysm = System(ctx, 4, "fp64", w["pos"], w["cell"], 4.0, 5.0)
    for st in ("XY", "TU", "Z", "Q", "W"):
        sysm.set_stage_kernel(st, "tensor-tile" if st == digits else other)
    sysm.set_mirror(mirror)
    sysm.profile(True)
    vals = [to_dev(M["val"], torch.float64, ctx.device) for M in (S, H, L)]
    for grad in (True, False):
        out, G, GN = sysm.energy_grad(*vals, grad=grad, grad_ne=True)
        assert abs(out[0, 0].item() - ref["E"]) <= 1e-12 * abs(ref["E"])
        assert abs(out[0, 1].item() - ref["Ne"]) <= 1e-12 * abs(ref["Ne"])
        assert rel_fro(GN.cpu().numpy(), ref["GN"]) <= 1e-13
        if grad:
            assert rel_fro(G.cpu().numpy(), ref["G"]) <= 1e-13
            assert all(v > 0 for v in sysm.stage_ms().values())
    assert ctx.device_status() == 0


def test_each_order_of_digits(ctx):
    """Rows of A with one digit per element, of order s, and columns of B with one of order t: products with s + t <= 5
    are exact, those of 6 and 7 are added in units of 2^-6 of order 5 (2^-58 here), so no order is missing or at a
    wrong place.  The largest elements, of the scales, meet zeros in these rows and columns, and are met in others (A's
    at inner index 0, B's at 1), so that the digits are kept."""
    rng = np.random.default_rng(2)
    n = 6
    a, b = np.zeros((4 * n, 4 * n)), np.zeros((4 * n, 4 * n))
    da, db = (rng.integers(-60, 61, size=(7, 4 * n - 2)) for _ in "ab")
    for s in range(7):  # the largest is 1: digit s has the weight 2^(-6 - 8 s)
        a[s, 0], a[s, 2:] = 1.0, da[s] * 2.0 ** (-6 - 8 * s)
        b[1, s], b[2:, s] = 1.0, db[s] * 2.0 ** (-6 - 8 * s)
    b[0, 10] = a[10, 1] = 1.0
    P = Pattern.build(ctx, np.random.default_rng(0).uniform(0, 5.0, size=(n, 3)), np.array([30.0, 30.0, 30.0]), 14.9)
    blocks = [np.ascontiguousarray(v.reshape(n, 4, n, 4).transpose(0, 2, 1, 3)).reshape(n * n, 4, 4) for v in (a, b)]
    plan = Plan(ctx, P, P, P)
    plan.set_kernel("tensor-tile")
    C = plan.multiply(*(to_dev(v, torch.float64, ctx.device) for v in blocks)).cpu().numpy()
    C = C.reshape(n, n, 4, 4).transpose(0, 2, 1, 3).reshape(4 * n, 4 * n)
    want = (da @ db.T) * 2.0 ** (-12.0 - 8.0 * np.add.outer(np.arange(7), np.arange(7)))
    order = np.add.outer(np.arange(7), np.arange(7))
    C = C[:7, :7]
    assert np.array_equal(C[order <= 5], want[order <= 5])
    low = (order == 6) | (order == 7)
    assert np.all(np.abs(C[low] - want[low]) <= 2.0 ** -59) and np.abs(want[order == 7]).min() > 2.0 ** -58
    assert np.all(C[order > 7] == 0.0)  # not formed


@pytest.mark.parametrize("nsf", [4, 9])
@pytest.mark.parametrize("spread", [10, 60, 300])
def test_norms_of_basis_functions_change_no_bit(ctx, nsf, spread):
    """S -> D S D, H -> D H D, L -> D^-1 L D^-1 with powers of two and S_kk = 1 before: the digits are those of the
    normalised functions, so E, N_e and the traces have the same bits, and dE/dL and dN_e/dL with D taken out."""
    rng = np.random.default_rng(nsf)
    from synth import si_diamond_positions, sym_block_values
    pos, cell = si_diamond_positions(2, rng)
    pos, r = np.ascontiguousarray(pos[:43]), (4.0, 6.0)
    pat = {k: oracle.pattern(pos, cell, c) for k, c in (("S", r[0]), ("H", r[0]), ("L", r[1]))}
    M = {k: oracle.csr(*pat[k], sym_block_values(*pat[k], pos, cell, nsf, k, rng)) for k in "SHL"}
    d = 2.0 ** np.round(spread * rng.uniform(-0.5, 0.5, size=(pos.shape[0], nsf)))
    got = []
    for dd in (np.ones_like(d), d):
        sysm = System(ctx, nsf, "fp64", pos, cell, *r)
        out, G, GN = sysm.energy_grad(*(to_dev(_rescaled(M[k], dd, p), torch.float64, ctx.device) for k, p in
                                        (("S", 1.0), ("H", 1.0), ("L", -1.0))), grad_ne=True)
        got.append([out.cpu().numpy()] + [_rescaled(dict(M["L"], val=g.cpu().numpy()), dd, -1.0) for g in (G, GN)])
    for x, y in zip(*got):
        assert np.array_equal(x, y)
    assert ctx.device_status() == 0


@pytest.mark.parametrize("bad", [0.0, np.nan, np.inf])
@pytest.mark.parametrize("zero", ["a", "b", "both", "some"])
def test_zero_rows_and_columns(ctx, zero, bad):
    """Operands of zeros, whole or in part: zeros against finite elements, NaN against others, as term by term."""
    rng = np.random.default_rng(3)
    P = Pattern.build(ctx, rng.uniform(0, 9.0, size=(42, 3)), np.array([20.0, 20.0, 20.0]), 6.0)
    v = {k: rng.standard_normal((P.nnzb, 4, 4)) for k in "ab"}
    rows = np.repeat(np.arange(42), np.diff(P.row_ptr.cpu().numpy()))
    for k in "ab":
        if zero in (k, "both"):
            v[k][:] = 0.0
        elif zero == "some":
            v[k][rows % 3 == 1] = 0.0
            v[k][P.col.cpu().numpy() % 5 == 2] = 0.0
            v[k][:, 2] = 0.0
    if bad != 0.0:
        v["a"][7, 1, 2] = bad
        v["b"][100, 0, 3] = bad
    out = {}
    for kernel in ("triples", "tensor-tile"):
        plan = Plan(ctx, P, P, P, trans_b=True)
        plan.set_kernel(kernel)
        out[kernel] = plan.multiply(*(to_dev(v[k], torch.float64, ctx.device) for k in "ab")).cpu().numpy()
    ref, C = out["triples"], out["tensor-tile"]
    assert np.array_equal(np.isnan(ref), np.isnan(C)) and np.array_equal(ref == 0.0, C == 0.0)
    fine = np.isfinite(ref)
    assert np.array_equal(ref[~fine & ~np.isnan(ref)], C[~fine & ~np.isnan(ref)])
    assert np.linalg.norm(C[fine] - ref[fine]) <= 1e-14 * np.linalg.norm(ref[fine])
    assert ctx.device_status() == 0


@pytest.mark.parametrize("nsf", [4, 9])
@pytest.mark.parametrize("unused", ["one", "all but one", "all", "diagonal only"])
def test_functions_that_l_does_not_use(ctx, nsf, unused):
    """Rows and columns of L that are zero (or only its diagonal element is): E, N_e, G and dN_e/dL of the oracle; a NaN of
    H at such a function still reaches E and G."""
    rng = np.random.default_rng(nsf)
    from synth import si_diamond_positions, sym_block_values
    pos, cell = si_diamond_positions(2, rng)
    pos, r = np.ascontiguousarray(pos[:43]), (4.0, 6.0)
    pat = {k: oracle.pattern(pos, cell, c) for k, c in (("S", r[0]), ("H", r[0]), ("L", r[1]))}
    M = {k: oracle.csr(*pat[k], sym_block_values(*pat[k], pos, cell, nsf, k, rng)) for k in "SHL"}
    rows = np.repeat(np.arange(43), np.diff(M["L"]["rp"]))
    L = M["L"]["val"]
    dead = {"one": [2], "all but one": list(range(1, nsf)), "all": list(range(nsf)), "diagonal only": []}[unused]
    L[:, dead, :] = 0.0
    L[:, :, dead] = 0.0
    if unused == "diagonal only":
        L[np.ix_(rows == M["L"]["col"], [1], [1])] = 0.0
    ref = oracle.lnv_energy_grad(pos, cell, *r, M["S"], M["H"], M["L"], grad=True, grad_ne=True)
    sysm = System(ctx, nsf, "fp64", pos, cell, *r)
    vals = [to_dev(M[k]["val"], torch.float64, ctx.device) for k in "SHL"]
    out, G, GN = sysm.energy_grad(*vals, grad_ne=True)
    assert abs(out[0, 0].item() - ref["E"]) <= 1e-12 * abs(ref["E"])
    assert abs(out[0, 1].item() - ref["Ne"]) <= 1e-12 * abs(ref["Ne"])
    assert rel_fro(G.cpu().numpy(), ref["G"]) <= 1e-13
    assert rel_fro(GN.cpu().numpy(), ref["GN"]) <= 1e-13
    vals[1][0, 2, 2] = float("nan")
    out, G = sysm.energy_grad(*vals)
    assert torch.isnan(out[0, 0]) and torch.isnan(G).any() and not torch.isnan(out[0, 1])
    assert ctx.device_status() == 0

"""The order in which the listed triples' items are taken, on patterns with one long row beside short ones (groups of
rows that fit shared memory and one that does not): the same sums as the push kernel."""
import numpy as np
import pytest
import torch

from paper_0911_3584_gb300 import Context, Pattern, Plan

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("sym_c", [False, True])
@pytest.mark.parametrize("n", [1, 3, 4, 5, 2000, 8192, 9000])
def test_arrow_patterns(cuda_device, n, sym_c):
    ctx = Context(cuda_device)
    # row n // 2 and column n // 2 full, and the diagonal
    h = n // 2
    rows = [np.unique([h, i]) if i != h else np.arange(n) for i in range(n)]
    rp = np.cumsum([0] + [r.size for r in rows])
    P = Pattern.from_csr(ctx, torch.from_numpy(rp), torch.from_numpy(np.concatenate(rows).astype(np.int32)))
    gen = torch.Generator(device=cuda_device).manual_seed(n)
    A, B = (torch.randn((P.nnzb, 4, 4), generator=gen, dtype=torch.float64, device=cuda_device) for _ in "ab")
    if sym_c:  # A A^T is symmetric
        B = A
        plans = [Plan(ctx, P, P, P, trans_b=True, sym_c=True) for _ in range(2)]
    else:
        plans = [Plan(ctx, P, P, P) for _ in range(2)]
    plans[0].set_kernel("triples")
    plans[1].set_kernel("push")
    C, ref = (p.multiply(A, B) for p in plans)
    assert (C - ref).norm() <= 1e-13 * ref.norm()
    assert torch.equal(C, plans[0].multiply(A, B))

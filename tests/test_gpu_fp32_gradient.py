"""The gradient's combination 6 (U + U^T) - 4 (Q^T + W + Q) of FP32 products."""
import numpy as np
import pytest
import torch

from paper_0911_3584_gb300 import Context, System

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx(cuda_device):
    return Context(cuda_device)


@pytest.mark.parametrize("nsf", [1, 2, 4, 9])
@pytest.mark.parametrize("h,l", [
    (1.5 * 2.0 ** 126, 1.0 - 2.0 ** -10),   # 4 U overflows, G does not
    (-1.99 * 2.0 ** 126, 1.0 - 2.0 ** -20), (2.0 ** 127, 1.0), (1.7 * 2.0 ** 127, 1.0 + 2.0 ** -23),
    (0.3, 1.0 - 2.0 ** -23), (0.3, 1.0 + 2.0 ** -22), (1e-30, 1.0 - 2.0 ** -12), (3e-38, 0.7), (0.7, 0.3)])
def test_fp32_gradient_is_combined_in_more_than_fp32(ctx, nsf, h, l):
    """One atom, one function that is not zero: dE/dL = 6 (U + U^T) - 4 (Q^T + W + Q) in FP64 of the FP32 products
    U = l h, Q = h l^2, W = l (l h), rounded once, also where terms cancel or 4 U leaves the range of FP32."""
    f = np.float32
    h, l = f(h), f(l)
    u, q = f(l * h), f(h * f(l * l))
    w = f(l * u)
    want = f(6.0 * (2.0 * np.float64(u)) - 4.0 * (2.0 * np.float64(q) + np.float64(w)))
    sysm = System(ctx, nsf, "fp32", np.zeros((1, 3)) + 1.0, [40.0, 40.0, 40.0], 4.0, 5.0)
    m = {k: torch.zeros((1, nsf, nsf), dtype=torch.float32, device=ctx.device) for k in "SHL"}
    m["S"][0, 0, 0], m["H"][0, 0, 0], m["L"][0, 0, 0] = 1.0, float(h), float(l)
    _, G = sysm.energy_grad(m["S"], m["H"], m["L"])
    assert np.isfinite(want)
    assert G[0, 0, 0].item() == want, (G[0, 0, 0].item(), want, u, q, w)


@pytest.mark.parametrize("nsf", [1, 4])
@pytest.mark.parametrize("h", [1.9 * 2.0 ** 127, -1.9 * 2.0 ** 127, float("inf"), float("nan")])
def test_fp32_gradient_that_leaves_the_range(ctx, nsf, h):
    """G = 12 h (l - l^2) beyond the range of FP32 is infinite, of its sign; NaN and infinite terms give NaN."""
    sysm = System(ctx, nsf, "fp32", np.zeros((1, 3)) + 1.0, [40.0, 40.0, 40.0], 4.0, 5.0)
    m = {k: torch.zeros((1, nsf, nsf), dtype=torch.float32, device=ctx.device) for k in "SHL"}
    m["S"][0, 0, 0], m["H"][0, 0, 0], m["L"][0, 0, 0] = 1.0, h, 0.5
    _, G = sysm.energy_grad(m["S"], m["H"], m["L"])
    want = np.copysign(np.inf, h) if np.isfinite(h) else np.nan
    assert np.array_equal(G[0, 0, 0].item(), want, equal_nan=True)

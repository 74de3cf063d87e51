"""The kernels that an FP32 system with 4 x 4 blocks begins with: the faster of the listed triples and the half-width
row groups (times beside the rule in mult.cu)."""
import numpy as np
import pytest

from paper_0911_3584_gb300 import Context, System
from synth import si_diamond_positions

pytestmark = pytest.mark.gpu

T, G = "triples", "group-pipe-half"


@pytest.mark.parametrize("ncell,want", [
    (1, dict(XY=T, TU=T, Z=T, Q=T, W=T)),
    (2, dict(XY=T, TU=T, Z=T, Q=T, W=T)),
    (3, dict(XY=T, TU=T, Z=G, Q=T, W=T)),   # W 66 us against 101
    (4, dict(XY=T, TU=G, Z=G, Q=G, W=T)),   # W 256 against 283
    (5, dict(XY=T, TU=G, Z=G, Q=G, W=G))])
def test_first_kernels_of_cubic_cells(cuda_device, ncell, want):
    pos, cell = si_diamond_positions(ncell, np.random.default_rng(0))
    assert System(Context(cuda_device), 4, "fp32", pos, cell, 6.6, 8.0).stage_kernels() == want


def test_first_kernels_of_a_batch(cuda_device):
    """Many small systems: few hits in X = LS although there are many triples (109 us against 131)."""
    cells = [si_diamond_positions(n, np.random.default_rng(n)) for n in (2, 2, 2, 2, 3, 3)]
    off = np.cumsum([0] + [p.shape[0] for p, _ in cells])
    sysm = System(Context(cuda_device), 4, "fp32", np.concatenate([p for p, _ in cells]), [c for _, c in cells], 6.6, 8.0,
                  seg_off=off)
    assert sysm.stage_kernels() == dict(XY=T, TU=G, Z=G, Q=G, W=T)

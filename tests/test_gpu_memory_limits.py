"""FP64 systems whose digits do not fit beside the intermediates (a shim in front of the runtime's cudaMemGetInfo says
what is free): they run without digits in the workspace that this takes, and are refused nothing."""
import os
import shutil
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SHIM = r"""
#define _GNU_SOURCE
#include <dlfcn.h>
#include <stddef.h>
static size_t says = 0;
void shim_free(size_t n) { says = n; }  /* what is free (0: the truth) */
int cudaMemGetInfo(size_t *f, size_t *t)
{
    static int (*real)(size_t *, size_t *);
    if (!real) real = (int (*)(size_t *, size_t *))dlsym(RTLD_NEXT, "cudaMemGetInfo");
    int e = real(f, t);
    if (says) *f = says;
    return e;
}
"""

CHILD = r"""
import ctypes, sys
import numpy as np, torch
import oracle
from paper_0911_3584_gb300 import Context, System
from synth import si_diamond_positions, sym_block_values
from tests.gpu_util import rel_fro, to_dev
shim = ctypes.CDLL(sys.argv[1])
shim.shim_free.argtypes = [ctypes.c_size_t]
dev = torch.device("cuda:0")
ctx = Context(dev)
for nsf, tensor in ((4, "tensor-tile"), (9, "tensor9")):
    rng = np.random.default_rng(nsf)
    pos, cell = si_diamond_positions(2, rng)
    pat = {k: oracle.pattern(pos, cell, r) for k, r in (("S", 4.0), ("H", 4.0), ("L", 5.0))}
    M = {k: oracle.csr(*pat[k], sym_block_values(*pat[k], pos, cell, nsf, k, rng)) for k in "SHL"}
    ref = oracle.lnv_energy_grad(pos, cell, 4.0, 5.0, M["S"], M["H"], M["L"], grad=True, grad_ne=True)
    vals = [to_dev(M[k]["val"], torch.float64, dev) for k in "SHL"]
    need = None
    for free in (0, 0, -1):
        shim.shim_free(need + free if need else 0)
        sysm = System(ctx, nsf, "fp64", pos, cell, 4.0, 5.0)
        shim.shim_free(0)
        size = sysm.workspace_size(True)
        if need is None:
            need, full = size + 2 * sum(v.numel() * 8 for v in vals[1:]), size
        assert (set(sysm.stage_kernels().values()) == {tensor}) == (free == 0), (nsf, free, sysm.stage_kernels())
        assert (size == full) == (free == 0)
        for pin in (False, True):
            if pin:  # outside the workspace then
                sysm.set_stage_kernel("Z", tensor)
            ws = torch.empty(sysm.workspace_size(True), dtype=torch.uint8, device=dev)
            out, G, GN = sysm.energy_grad(*vals, grad_ne=True, workspace=ws)
            assert abs(out[0, 0].item() - ref["E"]) <= 1e-12 * abs(ref["E"])
            assert abs(out[0, 1].item() - ref["Ne"]) <= 1e-12 * abs(ref["Ne"])
            assert rel_fro(G.cpu().numpy(), ref["G"]) <= 1e-13
            assert rel_fro(GN.cpu().numpy(), ref["GN"]) <= 1e-13
    print(nsf, "workspace with digits", full, "without", size, flush=True)
"""


def test_systems_without_room_for_digits(cuda_device, tmp_path):
    gcc = shutil.which("gcc") or shutil.which("cc")
    if not gcc:
        pytest.skip("no C compiler")
    (tmp_path / "shim.c").write_text(SHIM)
    shim = str(tmp_path / "shim.so")
    subprocess.run([gcc, "-shared", "-fPIC", "-o", shim, str(tmp_path / "shim.c"), "-ldl"], check=True)
    env = dict(os.environ, LD_PRELOAD=shim, PYTHONPATH=ROOT)
    r = subprocess.run([sys.executable, "-c", CHILD, shim], cwd=ROOT, env=env, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stdout[-2000:] + r.stderr[-3000:]

"""A lost copy in every precision of the march kernel: the launch whose bounded
waits expire and those after it write NaN, so that kpm_observables shows it in its
outputs, and rmft_iterate and rmft_iterate_batched report KPM_ETIMEDOUT.

M = 512: the last coefficient is then about 1e-10, so that a finite value written
in place of NaN, however large, would stay a finite result.  In child processes;
the copies are skipped, not failed, so nothing faults."""
import os
import subprocess
import sys

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

_CHILD = r"""
import sys
sys.path.insert(0, {root!r})
import torch
from paper_2212_05685_gb300 import build, inputs, kpm
build.build()
ctx = kpm.kpm_create(0)
nx, ny, M, prec, cells = 32, 16, 512, {prec}, {cells}
N = nx * ny
model = kpm.make_model(nx, ny)
phi = torch.empty(4 * N, dtype=torch.float64, device="cuda")
kpm.kpm_peierls_phases(ctx, model, phi)
w = inputs.Workload(nx, ny, 0.125, inputs.two_vortex(nx, ny), M)
seed = torch.tensor(inputs.vortex_seed(w), device="cuda")
fields = torch.empty(26 * N, dtype=torch.float64, device="cuda")
kpm.kpm_build_H(ctx, model, phi, seed, 0.0, fields)
ab = torch.empty(2, dtype=torch.float64, device="cuda")
kpm.kpm_bounds(ctx, model, fields, 0.01, ab)
opts = kpm.make_opts(M, prec)
ro = kpm.make_rmft_opts(w.n_target)
def observables():
    obs = torch.empty(26 * N, dtype=torch.float64, device="cuda")
    kpm.kpm_observables(ctx, model, opts, fields, ab, obs)
    st = ctx.lib.kpm_sync_status(ctx.handle, None)
    return st, obs
def iterate():
    mu = torch.zeros(1, dtype=torch.float64, device="cuda")
    return kpm.rmft_iterate(ctx, model, opts, ro, phi, seed.clone(), mu, 1, check=False)[0]
def batched():  # 1024 Nambu rows: FP32 cells of this size run the march kernel
    mu = torch.zeros(cells, dtype=torch.float64, device="cuda")
    return kpm.rmft_iterate_batched(ctx, [model] * cells, opts, [ro] * cells, [phi] * cells,
                                    [seed.clone() for _ in range(cells)], mu, 1, check=False)[0]
st, ref = observables()
assert st == kpm.KPM_OK and bool(torch.isfinite(ref).all())
kpm.kpm_inject_lost_copy(ctx, 1, 0.05)
st, bad = observables()
assert st == kpm.KPM_ETIMEDOUT, st
assert bool(torch.isnan(bad[:2 * N]).all()), "densities that are not NaN"
kpm.kpm_inject_lost_copy(ctx, 1, 0.05)
st = iterate()
assert st == kpm.KPM_ETIMEDOUT, ("iterate", st)
if cells:  # (double-float: refused by the batched call)
    kpm.kpm_inject_lost_copy(ctx, 1, 0.05)
    st = batched()
    assert st == kpm.KPM_ETIMEDOUT, ("batched", st)
kpm.kpm_inject_lost_copy(ctx, 0, 0.0)
st, again = observables()  # cleared: the same bits as before
assert st == kpm.KPM_OK and torch.equal(again, ref)
kpm.kpm_destroy(ctx)
print("lost-copy path ok")
"""


# the cells after a faulted one are NaN too: the batch reports the fault, not theirs
@pytest.mark.parametrize("prec,cells", [(0, 1), (0, 3), (1, 1), (1, 3), (2, 0)],
                         ids=["fp64", "fp64-3-cells", "fp32", "fp32-3-cells", "df64"])
def test_lost_copy_reads_as_nan(prec, cells):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    res = subprocess.run([sys.executable, "-c", _CHILD.format(root=root, prec=prec, cells=cells)], capture_output=True,
                         text=True, timeout=300)
    assert res.returncode == 0, res.stdout + res.stderr
    assert "lost-copy path ok" in res.stdout

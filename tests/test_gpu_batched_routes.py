"""rmft_iterate_batched takes FP32 cells of up to 640 Nambu rows through the
persistent recursion and larger ones through the march kernel, unless the scratch
budget does not hold their slabs: both routes, mixed and alone, give the
iterations of rmft_iterate (the moment sums and the recursion have the same
terms and order; 1e-12 as for the batch and the single cell elsewhere)."""
import numpy as np
import pytest

from paper_2212_05685_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def kpm():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2212_05685_gb300 import build, kpm
    build.build()
    return kpm


def _cell(kpm, ctx, nx, ny, k):
    w = inputs.Workload(nx, ny, 0.1 + 0.01 * k, inputs.two_vortex(nx, ny), 64, seed=k)
    model = kpm.make_model(nx, ny)
    phi = torch.empty(4 * nx * ny, dtype=torch.float64, device="cuda")
    kpm.kpm_peierls_phases(ctx, model, phi)
    return w, model, phi, torch.tensor(inputs.vortex_seed(w), device="cuda")


@pytest.mark.parametrize("shapes", [[(16, 20)], [(17, 19), (24, 24)], [(6, 4), (24, 24), (8, 8), (33, 11), (24, 24)],
                                    [(60, 8), (40, 40)]])
@pytest.mark.parametrize("M", [1, 2, 37])
@pytest.mark.parametrize("budget_mb", [0, 4])
def test_routes_follow_single_cells(kpm, shapes, M, budget_mb):
    ctx = kpm.kpm_create(0)
    if budget_mb:
        kpm.kpm_set_scratch_budget(ctx, budget_mb << 20)
    cells = [_cell(kpm, ctx, nx, ny, k) for k, (nx, ny) in enumerate(shapes)]
    params = [c[3].clone() for c in cells]
    ropts = [kpm.make_rmft_opts(c[0].n_target, tol=0.0) for c in cells]
    mu = torch.zeros(len(cells), dtype=torch.float64, device="cuda")
    opts = kpm.make_opts(M, kpm.KPM_FP32)
    for _ in range(2):  # the second call replays the graphs
        kpm.rmft_iterate_batched(ctx, [c[1] for c in cells], opts, ropts, [c[2] for c in cells], params, mu, 1)
    torch.cuda.synchronize()
    assert kpm.kpm_sync_status(ctx) == kpm.KPM_OK
    for k, c in enumerate(cells):
        one = kpm.kpm_create(0)
        p = c[3].clone()
        m = torch.zeros(1, dtype=torch.float64, device="cuda")
        for _ in range(2):
            kpm.rmft_iterate(one, c[1], opts, ropts[k], c[2], p, m, 1)
        torch.cuda.synchronize()
        assert np.max(np.abs((p - params[k]).cpu().numpy())) < 1e-12
        assert float(m.item()) == pytest.approx(float(mu[k].item()), abs=1e-12)
        kpm.kpm_destroy(one)
    kpm.kpm_destroy(ctx)

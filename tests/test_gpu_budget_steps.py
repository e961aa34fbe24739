"""How many steps per launch the default FP32 pass takes under scratch budgets that hold two slabs
of the full width but not four: two where four slabs of the narrower width still exceed L2,
else one on two full slabs.  Seen in the recursion's algorithmic bytes: 3 vectors a single
step (2 the first), 4 a launch of two steps (3 the first)."""
import pytest

from paper_2212_05685_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


# (lattice, budget in MB or 0 for the default, slab width, steps); D = 3400 and 6800
@pytest.mark.parametrize("nx,ny,budget_mb,width,steps", [
    (50, 34, 0, 3400, 2), (50, 34, 200, 3400, 1), (50, 34, 354, 3400, 2), (50, 34, 100, 1700, 1),
    (100, 34, 0, 6800, 2), (100, 34, 800, 3400, 2), (100, 34, 64, 567, 1)])
def test_steps_follow_the_width_that_runs(nx, ny, budget_mb, width, steps):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2212_05685_gb300 import build, kpm
    build.build()
    M = 9
    N = nx * ny
    out = []
    for budget in (0, budget_mb):
        ctx = kpm.kpm_create(0)
        if budget:
            kpm.kpm_set_scratch_budget(ctx, budget << 20)
        model = kpm.make_model(nx, ny)
        phi = torch.empty(4 * N, dtype=torch.float64, device="cuda")
        kpm.kpm_peierls_phases(ctx, model, phi)
        w = inputs.Workload(nx, ny, 0.125, inputs.two_vortex(nx, ny), M)
        p = torch.tensor(inputs.vortex_seed(w), device="cuda")
        mu = torch.zeros(1, dtype=torch.float64, device="cuda")
        _, st = kpm.rmft_iterate(ctx, model, kpm.make_opts(M, kpm.KPM_FP32), kpm.make_rmft_opts(w.n_target), phi, p, mu,
                                 1)
        out.append(p.cpu())
        kpm.kpm_destroy(ctx)
    ldv = -(-width // 16) * 16  # slabs advance by the padded width
    slabs = -(-2 * N // ldv)
    vector = 2 * N * ldv * 8
    vectors = 3 * (M - 1) - 1 if steps == 1 else 4 * (M - 1) // 2 - 1
    assert st.recursion_bytes == slabs * vectors * vector
    # the recursion has the same bits; the chemical potential's sums are FP64
    assert float((out[0] - out[1]).abs().max()) < 1e-12

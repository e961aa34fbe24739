"""The line between the persistent recursion and the march kernel in rmft_iterate_batched (FP32):
640 Nambu rows, 704 where a CTA's band is one lattice row of up to 46 sites or two of up to 28, 720 up to
11 sites wide (7: 672, 8: 640).  On both sides of it the cells follow rmft_iterate (1e-12, as for the batch elsewhere);
which route ran shows in the launches per iteration: one, or one a moment at least."""
import pytest

from paper_2212_05685_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,ny,persistent", [
    (20, 16, True), (17, 19, False), (28, 12, True), (29, 12, False), (22, 16, True), (23, 16, False), (41, 8, True),
    (46, 7, True), (47, 7, False), (45, 8, False), (11, 30, True), (11, 33, False), (12, 27, False), (5, 72, True),
    (5, 73, False), (8, 40, True), (8, 41, False), (7, 48, True), (7, 49, False), (9, 40, True), (50, 6, True), (33, 10, False)])
def test_route_and_results_at_the_line(nx, ny, persistent):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2212_05685_gb300 import build, kpm
    build.build()
    ctx, one = kpm.kpm_create(0), kpm.kpm_create(0)
    N, M = nx * ny, 21
    model = kpm.make_model(nx, ny)
    phi = torch.empty(4 * N, dtype=torch.float64, device="cuda")
    kpm.kpm_peierls_phases(ctx, model, phi)
    w = inputs.Workload(nx, ny, 0.1, inputs.two_vortex(nx, ny), M, seed=3)
    seed = torch.tensor(inputs.vortex_seed(w), device="cuda")
    ro, opts = kpm.make_rmft_opts(w.n_target, tol=0.0), kpm.make_opts(M, kpm.KPM_FP32)
    p, q = [seed.clone(), seed.clone()], seed.clone()
    mu, mu1 = torch.zeros(2, dtype=torch.float64, device="cuda"), torch.zeros(1, dtype=torch.float64, device="cuda")
    _, st = kpm.rmft_iterate_batched(ctx, [model] * 2, opts, [ro] * 2, [phi] * 2, p, mu, 1)
    kpm.rmft_iterate(one, model, opts, ro, phi, q, mu1, 1)
    assert (st[0].recursion_launches == 1) == persistent
    assert float((p[0] - q).abs().max()) < 1e-12 and float((p[1] - q).abs().max()) < 1e-12
    kpm.kpm_destroy(ctx)
    kpm.kpm_destroy(one)

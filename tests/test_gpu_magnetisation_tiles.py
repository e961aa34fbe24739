"""Values of the staggered magnetisation at the edges of the order-parameter kernel's 8 x 4 tiles: states
without bonds, whose exchange ratios are positive everywhere, with a magnetisation that differs from
site to site, so that a halo site read at the wrong place, or a site not written, shows.  Against
the oracle at the tolerance of the test of a larger lattice."""
import numpy as np
import pytest

from oracle import diagnostics, rmft

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,ny", [(2, 2), (3, 2), (2, 5), (7, 3), (8, 4), (9, 5), (15, 8), (16, 9), (17, 4), (33, 7)])
@pytest.mark.parametrize("bonds", [False, True])
def test_values_at_tile_edges(nx, ny, bonds):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2212_05685_gb300 import build, kpm
    build.build()
    ctx = kpm.kpm_create(0)
    N = nx * ny
    rng = np.random.default_rng(10 * nx + ny)
    mean, split = rng.uniform(0.40, 0.46, N), rng.uniform(0.02, 0.06, N) * np.where(rng.random(N) < 0.5, -1, 1)
    scale = 1e-3 if bonds else 0.0  # bonds too weak to turn a ratio negative
    chi = scale * (rng.standard_normal((2, 4, N)) + 1j * rng.standard_normal((2, 4, N)))
    F = scale * (rng.standard_normal((4, N)) + 1j * rng.standard_normal((4, N)))
    p = rmft.join(np.stack([mean + split, mean - split]), chi, F)
    model = kpm.make_model(nx, ny)
    phi = torch.empty(4 * N, dtype=torch.float64, device="cuda")
    kpm.kpm_peierls_phases(ctx, model, phi)
    d = torch.full((2 * N,), float("nan"), dtype=torch.float64, device="cuda")
    mg = torch.full((N,), float("nan"), dtype=torch.float64, device="cuda")
    kpm.kpm_order_parameters(ctx, model, phi, torch.tensor(p, device="cuda"), d, mg)
    torch.cuda.synchronize()
    want = diagnostics.staggered_magnetisation(rmft.Model(nx, ny, phi=phi.cpu().numpy().reshape(4, N)), p)
    assert np.isfinite(want).all() and np.min(np.abs(want)) > 1e-4
    assert np.max(np.abs(mg.cpu().numpy() - want)) < 1e-12 * max(1.0, np.max(np.abs(want)))
    kpm.kpm_destroy(ctx)

"""The order-parameter kernel works on 8 x 4 tiles with one site of halo: lattices
narrower than a tile and its halo, exact tiles, one site more and one less,
against the oracle at the tolerance of the test of a larger lattice."""
import numpy as np
import pytest

from oracle import diagnostics, rmft
from paper_2212_05685_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,ny", [(2, 2), (3, 2), (2, 5), (7, 3), (8, 4), (9, 5), (15, 8), (16, 9), (17, 4), (33, 7)])
def test_tile_edges(nx, ny):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2212_05685_gb300 import build, kpm
    build.build()
    ctx = kpm.kpm_create(0)
    N = nx * ny
    model = kpm.make_model(nx, ny)
    phi = torch.empty(4 * N, dtype=torch.float64, device="cuda")
    kpm.kpm_peierls_phases(ctx, model, phi)
    p = inputs.random_params(nx, ny, nx + ny, spin_split=0.02)
    d = torch.full((2 * N,), float("nan"), dtype=torch.float64, device="cuda")
    mg = torch.zeros(N, dtype=torch.float64, device="cuda")
    kpm.kpm_order_parameters(ctx, model, phi, torch.tensor(p, device="cuda"), d, mg)
    torch.cuda.synchronize()
    om = rmft.Model(nx, ny, phi=phi.cpu().numpy().reshape(4, N))
    got = d.cpu().numpy().reshape(N, 2)
    assert np.max(np.abs(got[:, 0] + 1j * got[:, 1] - diagnostics.physical_pairing(om, p))) < 1e-13
    assert np.array_equal(np.isnan(mg.cpu().numpy()), np.isnan(diagnostics.staggered_magnetisation(om, p)))
    kpm.kpm_destroy(ctx)

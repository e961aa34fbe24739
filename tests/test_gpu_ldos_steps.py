"""The diagonal-moment record of launches of several steps: the LDOS of all unit vectors on a lattice whose
slabs exceed L2 (100x34: two steps per launch) against narrow slabs, one step per launch.  The
record has the same bits, the FP64 contraction the same terms: 1e-12 of the largest value."""
import numpy as np
import pytest

from paper_2212_05685_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M", [2, 3, 8, 9])
def test_ldos_of_two_steps_per_launch(M):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2212_05685_gb300 import build, kpm
    build.build()
    ctx = kpm.kpm_create(0)
    nx, ny = 100, 34
    N = nx * ny
    model = kpm.make_model(nx, ny)
    phi = torch.empty(4 * N, dtype=torch.float64, device="cuda")
    kpm.kpm_peierls_phases(ctx, model, phi)
    fields = torch.empty(26 * N, dtype=torch.float64, device="cuda")
    kpm.kpm_build_H(ctx, model, phi, torch.tensor(inputs.random_params(nx, ny, 5), device="cuda"), 0.2, fields)
    ab = torch.empty(2, dtype=torch.float64, device="cuda")
    kpm.kpm_bounds(ctx, model, fields, 0.01, ab)
    omega = np.array([-0.8, -0.05, 0.0, 0.3])
    out = []
    for bw in (0, 400):
        ldos = torch.full((2 * len(omega) * N,), float("nan"), dtype=torch.float64, device="cuda")
        kpm.kpm_ldos(ctx, model, kpm.make_opts(M, kpm.KPM_FP32, block_width=bw), fields, ab, None, omega, ldos, 0.25, 0.05)
        assert kpm.kpm_sync_status(ctx) == kpm.KPM_OK
        out.append(ldos)
    assert float((out[0] - out[1]).abs().max()) < 1e-12 * float(out[1].abs().max())
    kpm.kpm_destroy(ctx)

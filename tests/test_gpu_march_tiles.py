"""KPM_FLAG_DOUBLE_STEP on lattice rows that two steps per launch split into tiles: the rings of the
fewest tiles that the threads allow do not fit shared memory at 26 sites (51, 52, 76 to 78, 101 to 104,
126 to 130, ...), so one more is taken; the pass runs two steps per launch and gives the bits
of single steps."""
import pytest

from paper_2212_05685_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,ny", [(50, 3), (51, 3), (52, 4), (53, 3), (78, 2), (104, 3), (130, 2), (156, 2), (182, 3)])
def test_double_step_of_every_tile_width(nx, ny):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2212_05685_gb300 import build, kpm
    build.build()
    ctx = kpm.kpm_create(0)
    N, M = nx * ny, 9
    model = kpm.make_model(nx, ny)
    phi = torch.empty(4 * N, dtype=torch.float64, device="cuda")
    kpm.kpm_peierls_phases(ctx, model, phi)
    w = inputs.Workload(nx, ny, 0.125, inputs.two_vortex(nx, ny), M)
    out = []
    for flags in (0, kpm.KPM_FLAG_DOUBLE_STEP):  # slabs of these sizes stay in L2: one step by default
        p = torch.tensor(inputs.random_params(nx, ny, 4), device="cuda")
        mu = torch.zeros(1, dtype=torch.float64, device="cuda")
        _, st = kpm.rmft_iterate(ctx, model, kpm.make_opts(M, kpm.KPM_FP32, flags=flags), kpm.make_rmft_opts(w.n_target),
                                 phi, p, mu, 1)
        assert st.recursion_launches == (M - 1) // (2 if flags else 1)
        out.append(p)
    assert torch.equal(out[0], out[1])
    kpm.kpm_destroy(ctx)

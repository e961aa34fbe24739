"""kpm_observables_noalloc where the march kernel's chunk of two slabs does not fit its 48 MiB and the one-step
kernels run: rows so wide that their chunk is 4 columns (224x224), and narrower chunks by cols_per_block
(100x500, refused at the default 16).  The recursion's numbers have the same bits as the march
kernel's and the FP64 sums the same terms: 1e-12 against kpm_observables."""
import pytest

from paper_2212_05685_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,ny,M,cols", [(224, 224, 3, 0), (224, 224, 2, 4), (224, 224, 2, 2), (100, 500, 3, 8),
                                          (100, 500, 2, 0)])
def test_one_step_kernels_of_the_allocation_free_call(nx, ny, M, cols):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2212_05685_gb300 import build, kpm
    build.build()
    ctx = kpm.kpm_create(0)
    N = nx * ny
    model = kpm.make_model(nx, ny)
    phi = torch.empty(4 * N, dtype=torch.float64, device="cuda")
    kpm.kpm_peierls_phases(ctx, model, phi)
    fields = torch.empty(26 * N, dtype=torch.float64, device="cuda")
    kpm.kpm_build_H(ctx, model, phi, torch.tensor(inputs.random_params(nx, ny, 5), device="cuda"), 0.2, fields)
    ab = torch.empty(2, dtype=torch.float64, device="cuda")
    kpm.kpm_bounds(ctx, model, fields, 0.01, ab)
    got, want = (torch.full((26 * N,), float("nan"), dtype=torch.float64, device="cuda") for _ in range(2))
    opts = kpm.make_opts(M, kpm.KPM_FP32, cols_per_block=cols)
    st = kpm.kpm_observables_noalloc(model, opts, fields, ab, got)
    if (nx, cols) == (100, 0):
        assert st == kpm.KPM_EINVAL
    else:
        assert st == kpm.KPM_OK
        kpm.kpm_observables(ctx, model, opts, fields, ab, want)
        torch.cuda.synchronize()
        assert float((got - want).abs().max()) < 1e-12
    kpm.kpm_destroy(ctx)

"""Recursion slabs of a context: which are allocated, kept and given back as passes of
different precision, steps per launch and width follow one another."""
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


def _cell(kpm, ctx, nx, ny):
    N = nx * ny
    model = kpm.make_model(nx, ny)
    phi = torch.empty(4 * N, dtype=torch.float64, device="cuda")
    kpm.kpm_peierls_phases(ctx, model, phi)
    fields = torch.empty(26 * N, dtype=torch.float64, device="cuda")
    kpm.kpm_build_H(ctx, model, phi, torch.tensor(inputs.random_params(nx, ny, 5), device="cuda"), 0.2, fields)
    ab = torch.empty(2, dtype=torch.float64, device="cuda")
    kpm.kpm_bounds(ctx, model, fields, 0.01, ab)
    return model, fields, ab


def _pass(kpm, ctx, cell, M, prec, **kw):
    model, fields, ab = cell
    obs = torch.full((26 * model.nx * model.ny,), float("nan"), dtype=torch.float64, device="cuda")
    kpm.kpm_observables(ctx, model, kpm.make_opts(M, prec, **kw), fields, ab, obs)
    assert kpm.kpm_sync_status(ctx) == kpm.KPM_OK
    return obs.cpu().numpy()


def _used():
    torch.cuda.synchronize()
    free, total = torch.cuda.mem_get_info()
    return total - free


def test_passes_in_turn_keep_their_slabs(kpm):
    """FP32 on four slabs of 370 MB (100x34: two steps per launch) and double-float on two
    of 655 MB (100x32), in turn: the device's memory in use stays where the first
    round of both put it (freeing one pass's slabs for the other's moves it by 169 MB)."""
    ctx = kpm.kpm_create(0)
    try:
        wide, other = _cell(kpm, ctx, 100, 34), _cell(kpm, ctx, 100, 32)
        ref = [_pass(kpm, ctx, wide, 5, kpm.KPM_FP32), _pass(kpm, ctx, other, 3, kpm.KPM_DF64)]
        level = _used()
        for _ in range(2):
            assert np.array_equal(_pass(kpm, ctx, wide, 5, kpm.KPM_FP32), ref[0])
            assert abs(_used() - level) < 16 << 20
            assert np.array_equal(_pass(kpm, ctx, other, 3, kpm.KPM_DF64), ref[1])
            assert abs(_used() - level) < 16 << 20
    finally:
        kpm.kpm_destroy(ctx)


def test_kept_slabs_stay_within_the_budget(kpm):
    """The same under a budget that holds each pass's slabs but not both together: what is
    held never exceeds it by more than the other scratch."""
    ctx = kpm.kpm_create(0)
    try:
        wide, other = _cell(kpm, ctx, 100, 34), _cell(kpm, ctx, 100, 32)
        budget = 1500 << 20
        kpm.kpm_set_scratch_budget(ctx, budget)
        empty = _used()
        first = None
        for _ in range(2):
            got = [_pass(kpm, ctx, wide, 5, kpm.KPM_FP32)]
            assert _used() - empty < budget + (64 << 20)
            got.append(_pass(kpm, ctx, other, 3, kpm.KPM_DF64))
            assert _used() - empty < budget + (64 << 20)
            first = first or got
            assert all(np.array_equal(a, b) for a, b in zip(got, first))
    finally:
        kpm.kpm_destroy(ctx)

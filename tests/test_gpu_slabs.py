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


def _room(nbytes):
    free, _ = torch.cuda.mem_get_info()
    if free < nbytes:
        pytest.skip("needs a device with that much free memory")


def test_two_slabs_where_four_do_not_fit_the_device(kpm):
    """220x220 under a budget above the device's memory: four slabs of 75 GB do not fit it,
    two do.  The pass runs one step per launch on two, with the bits of narrow slabs, and so does
    the next one."""
    torch.cuda.empty_cache()
    _room(200 << 30)
    ctx = kpm.kpm_create(0)
    try:
        cell = _cell(kpm, ctx, 220, 220)
        ref = _pass(kpm, ctx, cell, 3, kpm.KPM_FP32, block_width=4096)
        kpm.kpm_set_scratch_budget(ctx, 400 << 30)
        for flags in (0, kpm.KPM_FLAG_DOUBLE_STEP, 0):
            assert np.array_equal(_pass(kpm, ctx, cell, 3, kpm.KPM_FP32, flags=flags), ref)
            assert torch.cuda.mem_get_info()[0] > 100 << 30  # two slabs of 75 GB of 284
    finally:
        kpm.kpm_destroy(ctx)


def test_backward_after_a_pass_on_four_slabs(kpm):
    """220x196: the forward pass's four slabs of 60 GB fit the device, the backward pass's two
    vectors beside them do not; it runs on two of the slabs."""
    torch.cuda.empty_cache()
    _room(255 << 30)
    ctx = kpm.kpm_create(0)
    try:
        cell = model, fields, ab = _cell(kpm, ctx, 220, 196)
        go = torch.ones_like(fields)
        opts = kpm.make_opts(3, kpm.KPM_FP32)
        want, got = torch.empty_like(fields), torch.empty_like(fields)
        narrow = kpm.make_opts(3, kpm.KPM_FP32, block_width=8192)
        kpm.kpm_backward(ctx, model, narrow, fields, ab, go, 0.0, want, ckpt_every=kpm.KPM_REGENERATE)
        kpm.kpm_set_scratch_budget(ctx, 400 << 30)
        _pass(kpm, ctx, cell, 3, kpm.KPM_FP32)
        kpm.kpm_backward(ctx, model, opts, fields, ab, go, 0.0, got, ckpt_every=kpm.KPM_REGENERATE)
        assert kpm.kpm_sync_status(ctx) == kpm.KPM_OK
        # the sums over the columns are split at other places: FP32 rounding of their products
        assert float((got - want).abs().max()) < 1e-5 * float(want.abs().max())
    finally:
        kpm.kpm_destroy(ctx)

"""The FP32 march kernel (NS recursion steps per launch) at the edges of its
plans: the smallest lattices, rows that just fit one tile or just do not for one,
two and three steps, ragged last tiles, bands and slabs, odd site ranges, the
half pass, and every remainder of the order.

Its recursion vectors have the same bits for every plan, so passes that differ
only in steps per launch, bands and slabs are compared for equality; one of
them against the FP64 recursion within the FP32 tolerance of the other tests
(2e-5), which covers FP32 rounding over the order and nothing else.
"""
import numpy as np
import pytest

from paper_2212_05685_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def K():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2212_05685_gb300 import build, kpm
    build.build()
    ctx = kpm.kpm_create(0)
    yield kpm, ctx
    kpm.kpm_destroy(ctx)


def _cell(K, nx, ny):
    kpm, ctx = K
    N = nx * ny
    model = kpm.make_model(nx, ny)
    phi = torch.empty(4 * N, dtype=torch.float64, device="cuda")
    kpm.kpm_peierls_phases(ctx, model, phi)
    fields = torch.empty(26 * N, dtype=torch.float64, device="cuda")
    kpm.kpm_build_H(ctx, model, phi, torch.tensor(inputs.random_params(nx, ny, 5), device="cuda"), 0.2, fields)
    ab = torch.empty(2, dtype=torch.float64, device="cuda")
    kpm.kpm_bounds(ctx, model, fields, 0.01, ab)
    return model, fields, ab


def _pass(K, cell, M, prec=1, **kw):
    kpm, ctx = K
    model, fields, ab = cell
    obs = torch.full((26 * model.nx * model.ny,), float("nan"), dtype=torch.float64, device="cuda")
    om = torch.full((1,), float("nan"), dtype=torch.float64, device="cuda")
    kpm.kpm_observables(ctx, model, kpm.make_opts(M, prec, **kw), fields, ab, obs, om)
    assert kpm.kpm_sync_status(ctx) == kpm.KPM_OK
    return np.concatenate([obs.cpu().numpy(), om.cpu().numpy()])


# one tile up to 56 (one step), 28 (two) and 16 to 18 sites (three); 113 = 3 x 37 + 2
@pytest.mark.parametrize("nx,ny", [(2, 2), (2, 9), (3, 2), (17, 5), (19, 4), (28, 3), (29, 4), (31, 11), (56, 3),
                                   (57, 4), (58, 2), (113, 3)])
@pytest.mark.parametrize("M", [2, 3, 4, 24])
def test_plans_agree_bit_for_bit(K, nx, ny, M):
    kpm, _ = K
    cell = _cell(K, nx, ny)
    ref = _pass(K, cell, M)
    assert np.all(np.isfinite(ref))
    for kw in (dict(flags=kpm.KPM_FLAG_DOUBLE_STEP), dict(band_rows=1), dict(band_rows=max(1, ny - 1)),
               dict(block_width=40, flags=kpm.KPM_FLAG_DOUBLE_STEP, band_rows=2)):
        got = _pass(K, cell, M, **kw)
        assert np.array_equal(got[:-1], ref[:-1]), kw
        assert got[-1] == pytest.approx(ref[-1], rel=1e-12), kw
    if M == 24:
        assert np.max(np.abs(_pass(K, cell, M, 0)[:-1] - ref[:-1])) < 2e-5


@pytest.mark.parametrize("steps_flag", [0, 1])
def test_wide_slabs_take_two_and_three_steps(K, steps_flag):
    """100 x 34 sites: slabs above L2, so two steps per launch by default and three with the flag;
    against a pass of narrow slabs (one step per launch)."""
    kpm, ctx = K
    nx, ny, M = 100, 34, 9
    cell = _cell(K, nx, ny)
    wide = _pass(K, cell, M, flags=kpm.KPM_FLAG_DOUBLE_STEP * steps_flag)
    narrow = _pass(K, cell, M, block_width=1024)
    assert np.array_equal(wide[:-1], narrow[:-1])
    part = _pass(K, cell, M, site_begin=77, site_end=1234, flags=kpm.KPM_FLAG_DOUBLE_STEP * steps_flag)
    N = nx * ny
    for a, b in ((part[:N], wide[:N]), (part[N:2 * N], wide[N:2 * N])):
        assert np.array_equal(a[77:1234], b[77:1234])
        assert not a[:77].any() and not a[1234:].any()


def test_default_steps_shrink_to_the_budget(K):
    """A budget that holds two full slabs but not four: the default pass still runs, with the same bits."""
    kpm, _ = K
    nx, ny, M = 100, 34, 6
    cell = _cell(K, nx, ny)
    ref = _pass(K, cell, M)
    ctx = kpm.kpm_create(0)
    try:
        kpm.kpm_set_scratch_budget(ctx, 64 << 20)
        got = _pass((kpm, ctx), cell, M)
        assert np.array_equal(got[:-1], ref[:-1])
    finally:
        kpm.kpm_destroy(ctx)


@pytest.mark.parametrize("M", [1, 2, 3, 4, 5, 12])
@pytest.mark.parametrize("nx,ny,p,bw", [(2, 2, 2, 0), (12, 8, 4, 0), (12, 12, 3, 8), (60, 3, 3, 16)])
def test_probing_sums_of_every_order(K, nx, ny, p, bw, M):
    """FP32 probing keeps its moment sums two moments a launch, without the phase until the last
    moment: every remainder of the order, one and several slabs, against the FP64 pass of the same
    vectors (one-step kernels), within the FP32 tolerance of the other tests."""
    cell = _cell(K, nx, ny)
    kw = dict(block_width=bw, probe_p=p, probe_seed=3)
    assert np.max(np.abs(_pass(K, cell, M, 1, **kw)[:-1] - _pass(K, cell, M, 0, **kw)[:-1])) < 2e-5


@pytest.mark.parametrize("nx,ny", [(2, 2), (3, 5), (29, 4), (56, 3), (57, 4), (113, 2)])
@pytest.mark.parametrize("M", [2, 3, 9])
@pytest.mark.parametrize("prec", ["fp64", "df64"])
def test_fp64_and_double_float_plans(K, nx, ny, M, prec):
    """FP64 and double-float on the march kernel: the same bits for every band and slab, within
    1e-10 of the FP64 pass (double-float: about 48 bits, at most 9 steps of growth)."""
    kpm, _ = K
    P = kpm.KPM_FP64 if prec == "fp64" else kpm.KPM_DF64
    cell = _cell(K, nx, ny)
    ref = _pass(K, cell, M, P)
    for kw in (dict(band_rows=1), dict(band_rows=max(1, ny - 1)), dict(block_width=24, band_rows=2)):
        got = _pass(K, cell, M, P, **kw)
        assert np.array_equal(got[:-1], ref[:-1]), kw
    assert np.max(np.abs(_pass(K, cell, M, kpm.KPM_FP64)[:-1] - ref[:-1])) < 1e-10


@pytest.mark.parametrize("nx,ny", [(40, 40), (48, 48), (64, 32), (41, 43), (20, 128), (64, 64)])
def test_parts_of_a_slab_equal_slabs(K, nx, ny):
    """Slabs above L2 that run part after part through all their steps, against narrow slabs, whose
    launches have no parts."""
    cell = _cell(K, nx, ny)
    M = 8
    parts = _pass(K, cell, M)
    slabs = _pass(K, cell, M, block_width=400)
    assert np.array_equal(parts[:-1], slabs[:-1])
    N = nx * ny
    lo, hi = N // 7, N - 3
    part = _pass(K, cell, M, site_begin=lo, site_end=hi)
    assert np.array_equal(part[lo:hi], slabs[lo:hi])
    assert not part[:lo].any() and not part[hi:N].any()

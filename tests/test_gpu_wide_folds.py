"""The wide tiles' 8-bit counts hold whatever the lanes past the end of a row add
up to: those lanes sum bytes that nothing wrote (the rest of a stage behind a
clipped copy, padding of Y, workspace), up to fifteen counts per fold, and share
registers with valid sums.  Ragged last tiles, short delays, so that most windows
reach past their rows, and stages that hold chosen bytes beforehand; every row
equal to the narrow tile's."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

BAND = (1250.0, 1550.0, 81.92e-6)
MOST_FOLDS = 17  # 15 * 17 = 255


def _subband(lib, S, per, coarse, fine, n_t, top_dm):
    dms = top_dm / (coarse * fine) * np.arange(coarse * fine)
    return lib.Plan(S * per, *BAND, n_t, dms, [1], mode=lib.MODE_SUBBAND, n_subbands=S, coarse_dms=dms[::fine].copy())


def _step2_folds(S, per):
    """As the kernel makes them: two subbands at a time, eight per chunk."""
    every, folds, pending = 61440 // (255 * per), 0, 0
    for c in range(0, S, 8):
        left = min(8, S - c)
        while left:
            n = min(2, left)
            if pending + n > every:
                folds, pending = folds + 1, 0
            pending, left = pending + n, left - n
    return folds


def _fill_stages(lib, byte):
    """Leaves `byte` in the shared memory of every SM (windows of a constant input)."""
    import torch
    plan = lib.Plan(512, *BAND, 12500, 0.2 * np.arange(640), [1])
    cfg = plan.config
    cfg.brute = lib.DedispConfig(4, 16, 8, 1, 32, 0)
    plan.config = cfg
    x = torch.full((512, plan.pitch), byte, dtype=torch.uint8, device="cuda")
    lib.sps_dedisperse(plan, x, torch.empty((640, 12500), dtype=torch.int32, device="cuda"))


@pytest.mark.parametrize("S,per,n_t", [(64, 64, 12560), (48, 64, 12560), (32, 128, 12480), (36, 64, 12560),
                                       (34, 110, 12560), (128, 32, 12992)])
@pytest.mark.parametrize("byte", [0x05, 0x0c, 0x55, 0xf0])
def test_step_two(lib, S, per, n_t, byte):
    import torch
    plan = _subband(lib, S, per, 64, 32, n_t, 30.0)
    tile = plan.tiles()[0].step2
    wide = tile.as_tuple()[:2] == (8, 14)
    gen = torch.Generator(device="cuda").manual_seed(S)
    x = torch.randint(0, 256, (S * per, plan.pitch), dtype=torch.uint8, device="cuda", generator=gen)
    got = torch.full((plan.n_dms, n_t), -1, dtype=torch.int32, device="cuda")
    _fill_stages(lib, byte)
    lib.sps_dedisperse(plan, x, got)
    cfg = plan.config
    cfg.step2 = lib.DedispConfig(4, 8, 4, 1, 4, 0)
    plan.config = cfg
    want = torch.full((plan.n_dms, n_t), -2, dtype=torch.int32, device="cuda")
    lib.sps_dedisperse(plan, x, want)
    assert plan.status() == 0
    assert torch.equal(got, want)
    assert not wide or _step2_folds(S, per) <= MOST_FOLDS


def test_wide_step_two_where_its_counts_hold(lib):
    for S, per, kept in ((32, 48, True), (36, 64, True), (38, 64, False), (34, 120, True)):
        assert (_step2_folds(S, per) <= MOST_FOLDS) == kept
        assert (_subband(lib, S, per, 64, 32, 12560, 30.0).tiles()[0].step2.as_tuple()[:2] == (8, 14)) == kept


@pytest.mark.parametrize("C,step", [(4096, 0.002), (4096, 0.02), (3600, 0.004), (3240, 0.001)])
@pytest.mark.parametrize("byte", [0x04, 0x05])
def test_pass(lib, C, step, byte):
    import torch
    n_t, n_dms = 12560, 640
    plan = lib.Plan(C, *BAND, n_t, step * np.arange(n_dms), [1])
    assert plan.tiles()[0].brute.as_tuple()[:2] == (8, 14)
    gen = torch.Generator(device="cuda").manual_seed(C)
    x = torch.randint(0, 256, (C, plan.pitch), dtype=torch.uint8, device="cuda", generator=gen)
    ws = torch.full((plan.workspace_bytes,), byte, dtype=torch.uint8, device="cuda")
    got = torch.full((n_dms, n_t), -1, dtype=torch.int32, device="cuda")
    _fill_stages(lib, byte)
    lib.sps_dedisperse(plan, x, got, workspace=ws)
    cfg = plan.config
    cfg.brute = lib.DedispConfig(4, 16, 8, 1, 8, 2)
    plan.config = cfg
    want = torch.full((n_dms, n_t), -2, dtype=torch.int32, device="cuda")
    lib.sps_dedisperse(plan, x, want, workspace=ws)
    assert plan.status() == 0
    assert torch.equal(got, want)

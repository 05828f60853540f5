"""Which tiles the library picks, so that a test of a tile's results is known to
run that tile, and the forms that the tests of results alone do not reach."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

BAND = (1250.0, 1550.0, 81.92e-6)
WIDE = (8, 14)


def _plan(lib, C, n_t, n_dms, step):
    return lib.Plan(C, *BAND, n_t, step * np.arange(n_dms), [1])


def _subband(lib, S, per, coarse, fine, n_t, step=0.1):
    dms = step * np.arange(coarse * fine)
    return lib.Plan(S * per, *BAND, n_t, dms, [1], mode=lib.MODE_SUBBAND, n_subbands=S, coarse_dms=dms[::fine].copy())


def _step2(lib, plan, Y):
    import torch
    D = torch.full((plan.n_dms, plan.n_samples), -1, dtype=torch.int32, device="cuda")
    lib.sps_subband_step2(plan, Y, D)
    return D


def _narrow_step2(lib, plan, Y):
    cfg = plan.config
    cfg.step2 = lib.DedispConfig(4, 8, 4, 1, 4, 0)
    plan.config = cfg
    return _step2(lib, plan, Y)


def _y(plan, per, seed):
    import torch
    gen = torch.Generator(device="cuda").manual_seed(seed)
    return torch.randint(0, 255 * per + 1, plan.y_shape, dtype=torch.int32, device="cuda",
                         generator=gen).to(torch.int16).view(torch.uint16)


# brute force on quads: (channels, samples, trials, step) -> warps of the wide tile (0: the configured one), split
@pytest.mark.parametrize("shape,warps,split", [((1536, 3584, 2304, 0.2), 8, False), ((1536, 7013, 64, 0.2), 8, True),
                                               ((384, 3001, 300, 0.3), 8, True), ((389, 7013, 577, 0.31), 4, True),
                                               ((1536, 3001, 16, 0.2), 0, True), ((384, 12500, 700, 0.1), 0, False),
                                               ((5000, 1201, 40, 0.05), 0, True)])
def test_brute_tiles(lib, shape, warps, split):
    """Each form of the pass is known to run, and equals the single-channel kernel.  (384 channels x 700 trials: one
    wide round and four blocks more, 117 us, where the configured tile takes 99.)"""
    import torch
    plan = _plan(lib, *shape)
    tiles, splits, made = plan.tiles()
    assert tiles.brute.presum == 2 and not made
    assert (tiles.brute.warps_dm if tiles.brute.as_tuple()[:2] == WIDE else 0) == warps
    assert (splits > 1) == split
    gen = torch.Generator(device="cuda").manual_seed(shape[0])
    x = torch.randint(0, 256, (plan.channels, plan.pitch), dtype=torch.uint8, device="cuda", generator=gen)
    got = torch.full((plan.n_dms, plan.n_samples), -1, dtype=torch.int32, device="cuda")
    lib.sps_dedisperse(plan, x, got)
    cfg = plan.config
    cfg.brute = lib.DedispConfig(4, 16, 8, 1, 4, 0)
    plan.config = cfg
    want = torch.full((plan.n_dms, plan.n_samples), -2, dtype=torch.int32, device="cuda")
    lib.sps_dedisperse(plan, x, want)
    assert plan.status() == 0
    assert torch.equal(got, want)


def test_explicit_tiles_run_as_given(lib):
    plan = _plan(lib, 96, 2000, 40, 0.2)
    cfg = plan.config
    cfg.brute = lib.DedispConfig(4, 8, 4, 2, 16, 2)
    plan.config = cfg
    assert plan.tiles()[0].brute.as_tuple() == (4, 8, 4, 2, 16, 2)
    cfg.brute = lib.DedispConfig(4, 8, 4, 1, 8, 0)
    plan.config = cfg
    tiles, splits, made = plan.tiles()
    assert tiles.brute.as_tuple() == (4, 8, 4, 1, 8, 0) and splits == 1 and not made


@pytest.mark.parametrize("C,n_t,n_dms,step", [(100, 5001, 200, 0.5), (61, 4097, 70, 1.0), (64, 4096, 32, 2.0)])
def test_small_single_channel_plans_make_their_copies(lib, C, n_t, n_dms, step):
    plan = _plan(lib, C, n_t, n_dms, step)
    tiles, splits, made = plan.tiles()
    assert tiles.brute.presum == 0 and made


# subbands, channels per subband, coarse DMs, trials per coarse DM, samples -> warps along DM
@pytest.mark.parametrize("S,per,coarse,fine,n_t,warps", [(5, 120, 64, 32, 9001, 4), (17, 6, 128, 20, 4481, 3),
                                                         (32, 12, 96, 31, 14400, 4)])
def test_wide_step_two_runs_and_equals_narrow(lib, S, per, coarse, fine, n_t, warps):
    import torch
    plan = _subband(lib, S, per, coarse, fine, n_t)
    tile = plan.tiles()[0].step2
    assert tile.as_tuple()[:2] == WIDE and (tile.warps_dm, tile.warps_time) == (warps, 8 // warps)
    Y = _y(plan, per, S)
    got = _step2(lib, plan, Y)
    assert torch.equal(got, _narrow_step2(lib, plan, Y))
    assert plan.status() == 0


def test_short_runs_take_narrow_step_two(lib):
    """One or two warps along DM leave eight or four along time, whose stages do not fit two blocks an SM."""
    assert _subband(lib, 32, 12, 192, 7, 14400).tiles()[0].step2.as_tuple()[:2] != WIDE


@pytest.mark.parametrize("n_dms,n_t,decimate,threads", [(200, 55000, 1, 256), (4096, 20000, 1, 256), (4096, 12500, 1, 96),
                                                        (620, 4500, 0, 128), (620, 2000, 0, 64), (2000, 4500, 0, 64),
                                                        (100, 3000, 0, 256)])
def test_snr_threads(lib, n_dms, n_t, decimate, threads):
    """Rows of which an SM holds few keep their threads: decimation of 4096 rows of 55000 samples takes 379 us with
    96, 315 with 224; 620 rows of 4500 samples 18.7 us with 64, 14.8 with 128."""
    plan = lib.Plan(16, *BAND, n_t, 1e-3 * np.arange(n_dms), [1, 10], smoothing=decimate)
    assert plan.tiles()[0].snr.threads == threads


@pytest.mark.parametrize("tile", [(4, 8, 4, 1, 64, 1), (2, 8, 4, 1, 64, 1), (1, 8, 8, 1, 36, 1), (4, 8, 2, 1, 64, 1)])
def test_large_chunks(lib, tile):
    """Chunks of more than 16 series (one stage of them each), against the single-channel kernel."""
    import torch
    plan = _plan(lib, 389, 2011, 70, 0.05)
    gen = torch.Generator(device="cuda").manual_seed(9)
    x = torch.randint(0, 256, (389, plan.pitch), dtype=torch.uint8, device="cuda", generator=gen)
    out = []
    for t in (tile, (4, 8, 4, 1, 8, 0)):
        cfg = plan.config
        cfg.brute = lib.DedispConfig(*t)
        plan.config = cfg
        out.append(torch.full((70, 2011), -1, dtype=torch.int32, device="cuda"))
        lib.sps_dedisperse(plan, x, out[-1])
    assert plan.status() == 0
    assert torch.equal(*out)


def test_explicit_tiles_of_large_chunks_are_not_split_for_their_last_round(lib):
    """A block whose stage holds 32 pairs takes long to fill its ring: in three splits the pass of 1536 channels takes
    1006 us, in one 866."""
    plan = _plan(lib, 1536, 12500, 512, 0.1)
    cfg = plan.config
    cfg.brute = lib.DedispConfig(4, 8, 4, 1, 64, 1)
    plan.config = cfg
    assert plan.tiles()[1] == 1
    cfg.brute = lib.DedispConfig(8, 8, 4, 1, 16, 2)
    plan.config = cfg
    assert plan.tiles()[1] > 1

"""The wide tiles of the pre-summed pass, which take the default tile's place, and
the channel splits of small grids: every row equal to the single-channel
kernel's on the same plan, at the edges of the tiles (64 or 32 trials x 448
samples, chunks cut by window size, an odd last unit), of the 8-bit counts and of
the splits (added into rows that held other values)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

# channels, samples, trials, DM step, saturated input
CASES = [(41, 12501, 700, 0.05, False),    # 11 units, the last a single channel; rows of odd length
         (389, 7013, 577, 0.31, False),    # one trial past a tile, 293 samples in the last
         (384, 4480, 2048, 0.3, True),     # every lane at its bound, whole tiles only
         (4096, 1793, 2500, 0.02, True),   # the most channels: 255 counts
         (1536, 449, 11000, 0.02, False),  # one sample in the last time tile
         (1536, 3001, 16, 0.2, True),      # the 32-trial tile in sixteen splits, rows of odd length
         (389, 1003, 65, 0.2, False),      # splits with one trial in the last tile
         (1537, 450, 200, 0.3, False),     # an odd last unit in the last split
         (5000, 1201, 40, 0.05, True)]     # more channels than the counts hold: the default tile, split


@pytest.mark.parametrize("C,n_t,n_dms,step,full", CASES)
def test_wide_tile_equals_single_channel_kernel(lib, C, n_t, n_dms, step, full):
    import torch
    plan = lib.Plan(C, 1250.0, 1550.0, 81.92e-6, n_t, step * np.arange(n_dms), [1])
    assert plan.config.brute.presum == 2
    gen = torch.Generator(device="cuda").manual_seed(C)
    x = torch.randint(255 if full else 0, 256, (C, plan.pitch), dtype=torch.uint8, device="cuda", generator=gen)
    got = torch.full((n_dms, n_t), -1, dtype=torch.int32, device="cuda")
    lib.sps_dedisperse(plan, x, got)
    cfg = plan.config
    cfg.brute = lib.DedispConfig(4, 16, 8, 1, 4, 0)
    plan.config = cfg
    want = torch.full((n_dms, n_t), -2, dtype=torch.int32, device="cuda")
    lib.sps_dedisperse(plan, x, want)
    assert plan.status() == 0
    assert torch.equal(got, want)
    if full:
        assert int(got[0, 0]) == 255 * C


# subbands, channels per subband, coarse DMs, trials per coarse DM, samples, saturated
STEP2 = [(5, 120, 64, 32, 9001, True),    # the most channels per subband, an odd chunk, rows of odd length
         (17, 6, 128, 20, 4481, False),   # three warps along DM, the last with four trials
         (32, 12, 96, 7, 14400, False)]   # one warp along DM, runs shorter than its eight trials


@pytest.mark.parametrize("S,per,coarse,fine,n_t,full", STEP2)
def test_wide_step_two_equals_narrow(lib, S, per, coarse, fine, n_t, full):
    import torch
    dms = 0.1 * np.arange(coarse * fine)
    plan = lib.Plan(S * per, 1250.0, 1550.0, 81.92e-6, n_t, dms, [1], mode=lib.MODE_SUBBAND, n_subbands=S,
                    coarse_dms=dms[::fine].copy())
    gen = torch.Generator(device="cuda").manual_seed(S)
    Y = torch.randint(255 * per if full else 0, 255 * per + 1, plan.y_shape, dtype=torch.int32, device="cuda",
                      generator=gen).to(torch.int16).view(torch.uint16)
    got = torch.full((plan.n_dms, n_t), -1, dtype=torch.int32, device="cuda")
    lib.sps_subband_step2(plan, Y, got)
    cfg = plan.config
    cfg.step2 = lib.DedispConfig(4, 8, 4, 1, 4, 0)
    plan.config = cfg
    want = torch.full((plan.n_dms, n_t), -2, dtype=torch.int32, device="cuda")
    lib.sps_subband_step2(plan, Y, want)
    assert plan.status() == 0
    assert torch.equal(got, want)
    if full:
        assert int(got[0, 0]) == 255 * per * S


# channels, samples, trials, DM step, zapped channel or None: quads do not fit, so
# the default is the single-channel kernel
SINGLE = [(100, 5001, 200, 0.5, None), (61, 4097, 70, 1.0, 17), (64, 4096, 32, 2.0, 0)]


@pytest.mark.parametrize("C,n_t,n_dms,step,zap", SINGLE)
def test_copies_made_in_the_pass_brute(lib, C, n_t, n_dms, step, zap):
    """Small plans make the shifted copies of their windows in the pass; an
    explicit tile reads them from device memory."""
    import torch
    z = None if zap is None else [int(c == zap) for c in range(C)]
    plan = lib.Plan(C, 1250.0, 1550.0, 81.92e-6, n_t, step * np.arange(n_dms), [1], zap=z)
    assert plan.config.brute.presum == 0
    gen = torch.Generator(device="cuda").manual_seed(C)
    x = torch.randint(0, 256, (C, plan.pitch), dtype=torch.uint8, device="cuda", generator=gen)
    got = torch.full((n_dms, n_t), -1, dtype=torch.int32, device="cuda")
    lib.sps_dedisperse(plan, x, got)
    cfg = plan.config
    cfg.brute = lib.DedispConfig(4, 8, 4, 1, 8, 0)
    plan.config = cfg
    want = torch.full((n_dms, n_t), -2, dtype=torch.int32, device="cuda")
    lib.sps_dedisperse(plan, x, want)
    assert plan.status() == 0
    assert torch.equal(got, want)


@pytest.mark.parametrize("S,per,coarse,fine,n_t", [(7, 21, 40, 4, 6001), (32, 48, 64, 2, 3000), (3, 257, 9, 2, 1111)])
def test_copies_made_in_the_pass_step_one(lib, S, per, coarse, fine, n_t):
    import torch
    dms = 0.3 * np.arange(coarse * fine)
    plan = lib.Plan(S * per, 1250.0, 1550.0, 81.92e-6, n_t, dms, [1], mode=lib.MODE_SUBBAND, n_subbands=S,
                    coarse_dms=dms[::fine].copy())
    gen = torch.Generator(device="cuda").manual_seed(S)
    x = torch.randint(200, 256, (S * per, plan.pitch), dtype=torch.uint8, device="cuda", generator=gen)
    ys = []
    for tile in (None, (4, 8, 4, 1, 8, 0)):
        if tile:
            cfg = plan.config
            cfg.step1 = lib.DedispConfig(*tile)
            plan.config = cfg
        Y = torch.zeros(plan.y_shape, dtype=torch.int16, device="cuda").view(torch.uint16)
        lib.sps_subband_step1(plan, x, Y)
        ys.append(Y.view(torch.int16)[:, :, :plan.step1_samples])
    assert plan.status() == 0
    assert torch.equal(ys[0], ys[1])

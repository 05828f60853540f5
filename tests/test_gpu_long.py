"""Plans near the launch grid's limits (65535 blocks along its second dimension):
what the configured tile can run, the tile that the library picks in its place can
run too.  Rows of tens of millions of samples, and step two of very many short
rows, against the same sums in plain torch."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

BAND = (1250.0, 1550.0, 81.92e-6)


def _sum(x, delays, n_t):
    import torch
    out = torch.zeros(n_t, dtype=torch.int32, device=x.device)
    for c, d in enumerate(delays):
        out += x[c, d:d + n_t]
    return out


@pytest.mark.parametrize("mode,n_t,presum", [("brute", 30_000_000, 2), ("brute", 30_000_000, 0), ("subband", 20_000_000, 0)])
def test_long_rows(lib, mode, n_t, presum):
    import torch
    C, dms = 16, np.array([0.0, 0.7])
    kw = dict(mode=lib.MODE_SUBBAND, n_subbands=4, coarse_dms=[0.0]) if mode == "subband" else {}
    plan = lib.Plan(C, *BAND, n_t, dms, [1], **kw)
    if mode == "brute" and not presum:
        cfg = plan.config
        cfg.brute = lib.DedispConfig(4, 16, 8, 1, 16, 0)  # the default single-channel tile
        plan.config = cfg
    assert mode == "subband" or plan.config.brute.presum == presum
    gen = torch.Generator(device="cuda").manual_seed(n_t)
    x = torch.randint(0, 256, (C, plan.pitch), dtype=torch.uint8, device="cuda", generator=gen)
    D = torch.full((2, n_t), -1, dtype=torch.int32, device="cuda")
    lib.sps_dedisperse(plan, x, D)
    table = plan.delay_table()
    for i in range(2):
        assert torch.equal(D[i], _sum(x, table[i], n_t))
    assert plan.status() == 0


def test_step_two_of_many_short_rows(lib):
    import torch
    S, coarse, fine, n_t = 4, 20000, 32, 64
    dms = 1e-5 * np.arange(coarse * fine)
    plan = lib.Plan(2 * S, *BAND, n_t, dms, [1], mode=lib.MODE_SUBBAND, n_subbands=S, coarse_dms=dms[::fine].copy())
    gen = torch.Generator(device="cuda").manual_seed(1)
    Y = torch.randint(0, 511, plan.y_shape, dtype=torch.int32, device="cuda", generator=gen)
    D = torch.full((plan.n_dms, n_t), -1, dtype=torch.int32, device="cuda")
    lib.sps_subband_step2(plan, Y.to(torch.int16).view(torch.uint16), D)
    d2 = torch.from_numpy(plan.subband_tables()[1]).cuda().long()
    k = torch.arange(plan.n_dms, device="cuda") // fine
    t = torch.arange(n_t, device="cuda")
    want = sum(Y[k[:, None], s, d2[:, s, None] + t] for s in range(S))
    assert torch.equal(D, want.to(torch.int32))
    assert plan.status() == 0

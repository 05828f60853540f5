"""S/N rows of any length and place: the rows' aligned part is staged by one bulk
copy and the samples at either end by themselves, short rows take fewer threads,
and decimation up to twelve factors per pass.  The power-of-two kernel against
the general one (a width set with one more width), and rows that start anywhere
against the same rows on 16 bytes; all values bit for bit, since both forms take
S/N from the same exact integer moments."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

POW2 = [1, 2, 4, 8, 16, 32, 64]


def _table(lib, plan, D):
    import torch
    shape = (plan.n_widths, plan.n_dms)
    snr = torch.full(shape, -1.0, dtype=torch.float64, device="cuda")
    pt = torch.full(shape, -1, dtype=torch.int32, device="cuda")
    pv, best = pt.clone(), torch.full((4,), -1, dtype=torch.int32, device="cuda")
    lib.sps_snr(plan, D, snr, pt, pv, best)
    return snr, pt, pv, best


def _rows(n, n_t, seed):
    import torch
    gen = torch.Generator(device="cuda").manual_seed(seed)
    D = torch.randint(0, 255 * 96, (n, n_t), dtype=torch.int32, device="cuda", generator=gen)
    D[0] = 255 * 96                      # a constant row at its bound
    D[1, 0], D[2, n_t - 1] = 255 * 96, 255 * 96  # maxima at either end
    return D


@pytest.mark.parametrize("n_t", [64, 65, 66, 67, 1001, 4501, 7013, 12499])
@pytest.mark.parametrize("n", [20, 700])
def test_pow2_equals_general(lib, n_t, n):
    import torch
    D = _rows(n, n_t, n_t)
    dms = 0.001 * np.arange(n)
    a = _table(lib, lib.Plan(96, 1250.0, 1550.0, 81.92e-6, n_t, dms, POW2), D)
    b = _table(lib, lib.Plan(96, 1250.0, 1550.0, 81.92e-6, n_t, dms, [1, 2, 3, 4, 8, 16, 32, 64]), D)
    keep = [0, 1, 3, 4, 5, 6, 7]
    for x, y in zip(a[:3], b[:3]):
        assert torch.equal(x, y[keep])


@pytest.mark.parametrize("widths,smoothing", [(POW2, 0), ([1, 3, 10], 0), (list(range(1, 20, 2)), 1)])
@pytest.mark.parametrize("n_t", [64, 999, 5000])
def test_rows_anywhere(lib, n_t, widths, smoothing):
    import torch
    n = 40
    plan = lib.Plan(96, 1250.0, 1550.0, 81.92e-6, n_t, 0.001 * np.arange(n), widths, smoothing=smoothing)
    D = _rows(n, n_t, 7)
    want = _table(lib, plan, D)
    for off in (1, 2, 3):
        buf = torch.zeros(n * n_t + 4, dtype=torch.int32, device="cuda")
        view = buf[off:off + n * n_t].view(n, n_t)
        view.copy_(D)
        for x, y in zip(_table(lib, plan, view), want):
            assert torch.equal(x, y)

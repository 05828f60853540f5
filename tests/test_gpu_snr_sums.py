"""S/N sample sums of rows whose values leave no room in 32 bits: a thread's share
of a long row of near-saturated sums passes 2^32 (few threads per row, as
decimating plans of many trials take).  Against the two-pass S/N in float64, whose
own error over 56000 samples stays below 1e-10 relative; a sum that lost 2^32
moves S/N by far more."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("C,n_t,n_dms", [(32768, 56000, 160), (65536, 31999, 160), (131072, 9000, 700),
                                         (131072, 4500, 620)])
@pytest.mark.parametrize("widths,smoothing", [([1, 5, 40], 1), ([1, 3], 0), ([1, 2], 0)])
def test_sums_beyond_32_bits(lib, C, n_t, n_dms, widths, smoothing):
    import torch
    plan = lib.Plan(C, 1250.0, 1550.0, 81.92e-6, n_t, 1e-4 * np.arange(n_dms), widths, smoothing=smoothing)
    top = 255 * C
    gen = torch.Generator(device="cuda").manual_seed(C)
    D = torch.randint(top - top // 10, top + 1, (n_dms, n_t), dtype=torch.int32, device="cuda", generator=gen)
    shape = (len(widths), n_dms)
    snr = torch.full(shape, -1.0, dtype=torch.float64, device="cuda")
    pt, pv = (torch.full(shape, -1, dtype=torch.int32, device="cuda") for _ in range(2))
    lib.sps_snr(plan, D, snr, pt, pv)
    P = torch.nn.functional.pad(D.to(torch.int64).cumsum(1), (1, 0))
    for k, w in enumerate(widths):
        X = P[:, w::w] - P[:, :-w:w][:, :n_t // w] if smoothing else P[:, w:] - P[:, :-w]
        assert torch.equal(pv[k].long(), X.max(1).values)
        X = X.double()
        want = (X.max(1).values - X.mean(1)) / X.var(1, unbiased=False).sqrt()
        assert torch.allclose(snr[k], want, rtol=1e-8, atol=0)

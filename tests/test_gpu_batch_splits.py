"""Batches of few small beams split their channels as single searches do (in the
measure that the other beams leave SMs idle): every output equal to the single
search's, launch after launch, on rows that held other values."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


# beams as (channels, samples, trials, step)
@pytest.mark.parametrize("beams", [[(1536, 3001, 16, 0.2)], [(1536, 4000, 64, 0.3), (389, 1003, 65, 0.2)],
                                   [(384, 2500, 96, 0.2)] * 3, [(384, 5000, 512, 0.3), (1537, 450, 200, 0.3)]])
def test_batch_equals_search(lib, beams):
    import torch
    plans = [lib.Plan(C, 1250.0, 1550.0, 81.92e-6, n_t, step * np.arange(n), [1, 2, 4])
             for C, n_t, n, step in beams]
    assert any(p.tiles()[1] > 1 for p in plans)
    gen = torch.Generator(device="cuda").manual_seed(len(beams))
    xs = [torch.randint(0, 256, (p.channels, p.pitch), dtype=torch.uint8, device="cuda", generator=gen) for p in plans]
    want = [p.search(x) for p, x in zip(plans, xs)]
    batch = lib.Batch(plans, xs, branches=2)
    for fill in (-1, 7):
        for o in batch.outs:
            o["D"].fill_(fill)
        batch.launch()
        for p, o, w in zip(plans, batch.outs, want):
            for k in ("D", "snr", "peak_t", "peak_val", "best"):
                assert torch.equal(o[k], w[k]), k
            assert p.status() == 0
